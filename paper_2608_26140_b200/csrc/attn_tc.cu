// Bidirectional attention of many recomputed rows over the whole context (Section 4.3) on the
// 5th-generation tensor cores.  Three kernels share the scheme below: attention_tc_kernel (one CTA = 128
// query rows of one head; used when a request has at most 128 rows), attention_group_kernel (the same rows
// from several requests) and attention_tc2q_kernel (one CTA = 256 query rows), the last two described
// where they are defined.  Key/value tiles of 128 keys stream through shared
// memory by TMA (3-d tensor maps: positions past the context end and rows past the request's row count
// read as zero).
//
//   S = Q K^T    tcgen05.mma 128 x 128 x 16, both operands K-major, into a TMEM buffer
//   softmax      scaled max, exp2, running denominator; P is written as packed bf16 over the low
//                columns of its S buffer, so it never passes through shared memory
//   O += P V     tcgen05.mma 128 x 128 x 16, A = P read from tensor memory, B = V read in place as an
//                MN-major operand (token-major V rows are contiguous along the head dimension)
//
// One-tile kernel: sixteen softmax warps, four threads per query row (32 keys each), two S buffers: the
// S of tile j+1 is issued before the softmax of tile j is consumed, so tensor work overlaps the
// exponentials.  The running maximum used for the exponent is only raised (and O rescaled in
// TMEM) when the true maximum has grown by more than 2^8, which keeps P within bf16 range and
// makes rescales rare.  Every mbarrier wait is bounded (status flag kFlagWaitExpired on expiry).
// With two key sources (a cache shared by the batch + each request's private rows, Section 4.1) the
// private rows' tiles follow the cache's, and key masks tell which of the two serves a position.  When
// every request brings at most 64 rows (decode passes), two or four requests share one query tile
// (attention_group_kernel, below the one-tile kernel).
#include <climits>
#include <type_traits>
#include <cuda.h>

#include <mutex>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"
#include "tc_ptx.cuh"

namespace acache {

constexpr int AT_THREADS = 608;                  // warp 0: TMA, warp 1: S MMAs, warps 2-17: softmax (four threads per row), warp 18: PV MMAs
constexpr int AT_TILE = 128 * 128 * 2;           // 32 KB: a [128 x 128] bf16 tile as two 64-column panels
constexpr int AT_PANEL = 128 * 64 * 2;           // 16 KB
constexpr int AT_SLACK = 256;                    // the dynamic window starts 1024-aligned in practice; checked at run time
constexpr int AT_SMEM = 5 * AT_TILE + AT_SLACK + 256;   // Q, K x2, V x2 (P lives in tensor memory)
static_assert(AT_SMEM >= kAloneBytes);
constexpr float kRescaleGap = 8.f;               // log2 units

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar,
                                            uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const float (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]),
          "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]), "f"(v[16]), "f"(v[17]),
          "f"(v[18]), "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]), "f"(v[24]), "f"(v[25]), "f"(v[26]),
          "f"(v[27]), "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31])
        : "memory");
}
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 2^x on the FMA pipe for x <= ~8 (Cody-Waite: x = n + f with n = rint(x), |f| <= 0.5; a cubic for 2^f
// with relative error 7.5e-5, far below the bf16 rounding of P; n goes straight into the exponent).
// A quarter of the exponentials take this route so that the MUFU pipe is not the only one working.
__device__ __forceinline__ float poly_exp2(float x) {
    x = fmaxf(x, -126.f);
    const float t = x + 12582912.f;                 // 1.5 * 2^23: the low mantissa bits now hold rint(x)
    const float f = x - (t - 12582912.f);
    const float p = fmaf(fmaf(fmaf(0.05517146f, f, 0.24261086f), f, 0.69326097f), f, 0.9999281f);
    return __int_as_float(__float_as_int(p) + (__float_as_int(t) << 23));
}
// Barrier of 128 threads that also tells them whether any of them passes true.
__device__ __forceinline__ bool quarter_any(int barrier, bool pred) {
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, r;\n\t"
        "setp.ne.u32 p, %2, 0;\n\t"
        "barrier.cta.red.or.pred r, %1, 128, p;\n\t"
        "selp.u32 %0, 1, 0, r;\n\t}"
        : "=r"(any)
        : "r"(barrier), "r"((uint32_t)pred)
        : "memory");
    return any != 0;
}
// D += A B with A read from tensor memory (rows = TMEM lanes, two bf16 of consecutive K per 32-bit column)
__device__ __forceinline__ void tc_mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}
// The two products with D written only in the 32-lane quarters of `lanes` (bit q = quarter q).
__device__ __forceinline__ void tc_mma_lanes(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc, uint32_t lanes) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %6, %7, %8}, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"((lanes & 1u) - 1u), "r"(((lanes >> 1) & 1u) - 1u),
          "r"(((lanes >> 2) & 1u) - 1u), "r"(((lanes >> 3) & 1u) - 1u)
        : "memory");
}
__device__ __forceinline__ void tc_mma_ta_lanes(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t acc, uint32_t lanes) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %6, %7, %8}, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc), "r"((lanes & 1u) - 1u), "r"(((lanes >> 1) & 1u) - 1u),
          "r"(((lanes >> 2) & 1u) - 1u), "r"(((lanes >> 3) & 1u) - 1u)
        : "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
          "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// MN-major bf16 operand with the 128-byte swizzle: rows of the K index are 128 bytes (64 elements
// of the MN index), 8-row groups 1024 bytes apart (stride byte offset), and the next 64 elements
// of the MN index start one 16 KB panel further (leading byte offset).
__device__ __forceinline__ uint64_t smem_desc_mn_sw128(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(AT_PANEL >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

struct AttnTcArgs {
    void* o;                  // bf16 [B, n, H*d]
    int n, ctx_len, n_heads, n_kv_heads;
    float scale_log2e;
    uint32_t* status;
    // two key sources (shared storage + private rows, Section 4.1): after the cache's tiles come the tiles of
    // the fresh rows [B, n, Hkv, d]; pos_excl masks the cache positions those rows serve, row_keep the fresh
    // rows that do not serve their position (duplicates).  n_fresh_tiles = 0: the cache alone; pos_excl may then
    // still name cache positions that do not exist as keys (the DropNA layout of Section 5.3).
    int n_fresh_tiles, excl_words, keep_words, cache_shared;
    int kv_prefetch;          // two-query-tile kernel: K/V tiles requested into L2 ahead of the rings
    int group, batch;         // attention_group_kernel: requests per query tile, requests in all
    int split;                // one-tile kernels: CTAs (a cluster) per query tile, each over a part of the key tiles
    int n_items;              // one-tile kernels: query tiles over all heads and requests (or groups)
    const uint32_t* pos_excl;
    const uint32_t* row_keep;
    // Eq. 4-5 taken from this attention's own logits (two-query-tile kernel; the one-shot probe of Section 3.2): for the
    // query rows flagged in score_rowmask [B, rm_words] (bit i = compact row i is a masked position) the kernel keeps,
    // next to the softmax denominator, the same sum restricted to the affix keys, and after the last key tile walks the
    // affix key tiles once more with the product turned round (D = K Q^T: thread = key, columns = query rows), adding
    // exp2(s - reference) / denominator over the flagged rows.  score_partial [B, H, q_tiles, L]: per (head, 128-row
    // query tile) column sums, written only by tiles that hold flagged rows.
    const uint32_t* score_rowmask;
    float* score_partial;
    int rm_words, q_tiles, affix_start, affix_len;
    int score_norm_full;      // weight = 1 / the full denominator (Eq. 4 over every key) instead of the affix keys' share
};

// Wait for the two-query-tile kernel's threads whose hand-overs sit on the critical path of every key tile (the thread that
// issues the tensor-core instructions, the softmax threads waiting for S): no sleep between polls (the many-row attention
// went from 785 to 748 us on a 14 752-row layer; the one-tile kernel did not change); bounded like every wait.
__device__ __forceinline__ bool mbar_spin(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    for (uint32_t i = 0; i < (TC_WAIT_LIMIT << 4); ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 4095u) == 4095u && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

// A key tile of one query row's quarter (32 keys per thread): S from tensor memory at tS, P written back over its low columns, O
// at tO rescaled when the reference moves.  Four threads share a row; their warps (one lane quarter, one scheduler) meet at a vote
// every tile and only ever leave the loop together: a thread whose wait ran out (ok = false) skips its work and votes for the
// exchange, where all four learn of it and this returns false.  row_max: this row's entry of the first of four arrays, `stride` apart.
// The softmax is on the chain of every tile; with the maxima of all tiles exchanged through shared memory and one fp32 operation
// per element at a time it took 2000 cycles of a tile's 2600-3100 (maximum 280, 500 with masked keys; exchange 350; exponentials
// 1200-1300).  With the vote, masks applied once and packed fp32 arithmetic: attention of 1639 rows over 8288 keys 260 -> 235 us.
template <class WaitS, class WaitPrevious>
__device__ __forceinline__ bool softmax_tile(uint32_t keep, bool first, float scale_log2e, uint32_t tS, uint32_t tO, int c4, int vote,
                                             uint16_t* row_max, int stride, uint32_t p_full, float& m_use, float& l, bool& ok,
                                             WaitS wait_s, WaitPrevious wait_previous) {
    float sv[32];
    float mt = -INFINITY;
    if (ok && (ok = wait_s())) {
        tc_fence_after();
        // this thread's quarter row of S into registers, masked keys as -inf
        tc_ld32(tS + c4 * 32, sv);
        if (keep != 0xffffffffu) {
#pragma unroll
            for (int i = 0; i < 32; ++i) sv[i] = ((keep >> i) & 1u) ? sv[i] : -INFINITY;
        }
        float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int i = 0; i < 32; i += 2) m4[(i >> 1) & 3] = fmaxf(fmaxf(m4[(i >> 1) & 3], sv[i]), sv[i + 1]);
        mt = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * scale_log2e;
    }
    // The four threads of a row must use the same reference.  It moves on the first tile and seldom after; whether it
    // has to is one vote of the four warps that share these 32 rows, at the barrier that they need anyway (every
    // thread of a row must have read its S columns before P overwrites them).  A thread whose wait ran out votes too.
    bool raise = false;
    if (quarter_any(vote, !ok || mt - m_use > kRescaleGap)) {
        // all take the largest of the four quarter-row maxima rounded up to 16 significant bits (an upper bound is
        // all the exponent needs)
        uint32_t mb = __float_as_uint(mt);
        if ((mb & 0xFFFFu) && !(mb >> 31)) mb += 0x10000u;
        mb >>= 16;
        row_max[c4 * stride] = (uint16_t)mb;
        if (quarter_any(vote, !ok)) { ok = false; return false; }      // the four warps leave together
        mt = fmaxf(fmaxf(__uint_as_float((uint32_t)row_max[0] << 16), __uint_as_float((uint32_t)row_max[stride] << 16)),
                   fmaxf(__uint_as_float((uint32_t)row_max[2 * stride] << 16), __uint_as_float((uint32_t)row_max[3 * stride] << 16)));
        if (first) m_use = mt;
        else raise = mt - m_use > kRescaleGap;
    }
    if (__any_sync(0xffffffffu, raise)) {
        // O may only be touched once the P V of the tile before has completed
        if ((ok = wait_previous())) {
            tc_fence_after();
            const float f = raise ? fast_exp2(m_use - mt) : 1.f;
            float v[32];
            tc_ld32(tO + c4 * 32, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] *= f;
            tc_st32(tO + c4 * 32, v);
            tc_wait_st();
            l *= f;
            if (raise) m_use = mt;
        }
    }
    if (!ok) return true;
    // P overwrites the S buffer in tensor memory: 32 keys = 16 columns of two bf16 at column 16 c4
    // (every thread of the row has read its S columns: they all passed the vote above)
    const float neg = m_use > -INFINITY ? -m_use : 0.f;      // no key of the row has counted yet: all P are 0
    const float2 scale2 = make_float2(scale_log2e, scale_log2e), neg2 = make_float2(neg, neg);
    float2 l2a = make_float2(0.f, 0.f), l2b = l2a;
    uint32_t pk[16];
    auto exps = [&](auto all_kept) {
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
            const float2 xa = __ffma2_rn(make_float2(sv[i], sv[i + 1]), scale2, neg2);
            const float2 xb = __ffma2_rn(make_float2(sv[i + 2], sv[i + 3]), scale2, neg2);
            const float2 pa = make_float2(fast_exp2(xa.x), fast_exp2(xa.y));
            const float2 pb = make_float2(fast_exp2(xb.x), all_kept.value ? poly_exp2(xb.y) : fast_exp2(xb.y));
            l2a = __fadd2_rn(l2a, pa);
            l2b = __fadd2_rn(l2b, pb);
            pk[i >> 1] = pack_bf16(pa.x, pa.y);
            pk[(i >> 1) + 1] = pack_bf16(pb.x, pb.y);
        }
    };
    if (keep == 0xffffffffu) exps(std::true_type{});
    else exps(std::false_type{});
    tc_st16(tS + c4 * 16, pk);
    tc_wait_st();
    l += (l2a.x + l2a.y) + (l2b.x + l2b.y);
    tc_fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(p_full);
    return true;
}
// 32 columns of a finished row: O / l as bf16, 16 bytes a store.
__device__ __forceinline__ void store_o32(__nv_bfloat16* out, const float (&v)[32], float inv) {
#pragma unroll
    for (int k8 = 0; k8 < 4; ++k8) {
        const float* pv = v + k8 * 8;
        *reinterpret_cast<uint4*>(out + k8 * 8) =
            make_uint4(pack_bf16(pv[0] * inv, pv[1] * inv), pack_bf16(pv[2] * inv, pv[3] * inv),
                       pack_bf16(pv[4] * inv, pv[5] * inv), pack_bf16(pv[6] * inv, pv[7] * inv));
    }
}

// The cache's key tiles that hold a key for any of the requests [b0, b0 + n_req): tiles [x, y).  Private rows serve whatever
// lies outside the affix, so the tiles in front of it and behind it often hold none (a context of 2560 positions with 2048 affix
// rows: 4 of 20).  Where a cluster shares the key tiles they are all visited: most CTAs of it would gain nothing, and the look at the
// masks takes 1.5 us.  Called by all threads; lo_hi in shared memory holds (INT_MAX, 0) before the block's last barrier.
__device__ __forceinline__ int2 kept_tiles(const AttnTcArgs& a, int b0, int n_req, int* lo_hi) {
    const int n = (a.ctx_len + 127) / 128;
    if (!a.pos_excl) return make_int2(0, n);
    int first = INT_MAX, end = 0;                  // a word (32 positions of one request) per thread and round
    for (int i = threadIdx.x; i < n * 4 * n_req; i += blockDim.x) {
        const int r = i / (n * 4), w = i - r * n * 4, valid = a.ctx_len - w * 32;
        uint32_t in = valid >= 32 ? ~0u : (valid <= 0 ? 0u : (1u << valid) - 1u);
        if (w < a.excl_words) in &= ~__ldg(a.pos_excl + (int64_t)(b0 + r) * a.excl_words + w);
        if (in) {
            first = min(first, w >> 2);
            end = max(end, (w >> 2) + 1);
        }
    }
    first = __reduce_min_sync(0xffffffffu, first);
    end = __reduce_max_sync(0xffffffffu, end);
    if ((threadIdx.x & 31) == 0 && end > 0) {
        atomicMin(lo_hi, first);
        atomicMax(lo_hi + 1, end);
    }
    __syncthreads();
    const int lo = lo_hi[0], hi = lo_hi[1];
    return lo < hi ? make_int2(lo, hi) : make_int2(0, 0);
}
// Merge of a cluster's parts through distributed shared memory: every CTA leaves (reference, denominator) of its rows and its O as it
// is, laid out by the CTA that finishes the columns (128 / C each); behind one barrier that CTA scales the parts to the common
// reference and sums them in rank order.  (With the references met first and the parts scaled before they were laid out there
// was a barrier more: layer-step of 103 rows over 1024 keys 146.2 -> 145.7 us.)  The K and V stages are idle by now.  All threads pass the two cluster
// barriers, whatever happened before.  out: the row's 128 columns, null for a row that does not exist; any: this CTA had key
// tiles (else its O holds nothing).
__device__ __forceinline__ void merge_parts(uint32_t base, unsigned char* base_ptr, int C, int rank, bool softmax, bool any, int c4,
                                            int row, uint32_t tO, float m_use, float l, __nv_bfloat16* out) {
    float2* ml = reinterpret_cast<float2*>(base_ptr + AT_TILE + 4096);             // [128]
    const uint32_t parts = base + 2 * AT_TILE;                                     // [owner][column / 4][row][4] fp32
    const int width = 128 / C;
    __syncwarp();
    if (softmax) {
        if (c4 == 0) ml[row] = make_float2(m_use, l);
        tc_fence_after();
        float v[32];
        tc_ld32(tO + c4 * 32, v);
        const uint32_t dst = parts + ((c4 * 8 * 128 + row) << 4);                  // owners' columns lie one after the other
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 p = any ? make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + i * 2048), "f"(p.x), "f"(p.y), "f"(p.z), "f"(p.w) : "memory");
        }
    }
    __syncwarp();
    cluster_sync_all();
    if (softmax) {
        const int col = rank * width + c4 * (width >> 2);                          // width / 4 columns per thread
        const uint32_t ml_row = smem_u32(ml + row);
        float ref = -INFINITY, denom = 0.f, f[8], l_c[8];
        float4 u[8];
        const uint32_t src0 = parts + ((col >> 2) * 128 + row) * 16;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < C) {
                asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(f[c]), "=f"(l_c[c]) : "r"(mapa_u32(ml_row, c)) : "memory");
                asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                             : "=f"(u[c].x), "=f"(u[c].y), "=f"(u[c].z), "=f"(u[c].w) : "r"(mapa_u32(src0, c)) : "memory");
            }
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < C) ref = fmaxf(ref, f[c]);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < C) {
                f[c] = f[c] > -INFINITY ? fast_exp2(f[c] - ref) : 0.f;             // no key of the row has counted there: its part is 0
                denom += l_c[c] * f[c];
            }
        const float inv = 1.f / denom;
#pragma unroll 1
        for (int g4 = 0; g4 < width >> 4; ++g4) {
            if (g4 > 0) {
                const uint32_t src = src0 + g4 * 128 * 16;
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c < C)
                        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                                     : "=f"(u[c].x), "=f"(u[c].y), "=f"(u[c].z), "=f"(u[c].w) : "r"(mapa_u32(src, c)) : "memory");
            }
            float4 o = make_float4(__fmul_rn(u[0].x, f[0]), __fmul_rn(u[0].y, f[0]), __fmul_rn(u[0].z, f[0]), __fmul_rn(u[0].w, f[0]));
#pragma unroll
            for (int c = 1; c < 8; ++c)
                if (c < C) {
                    o.x += __fmul_rn(u[c].x, f[c]); o.y += __fmul_rn(u[c].y, f[c]);
                    o.z += __fmul_rn(u[c].z, f[c]); o.w += __fmul_rn(u[c].w, f[c]);
                }
            if (g4 + 1 == width >> 4) cluster_arrive();      // the last read: before the stores, which it would wait for
            if (out) *reinterpret_cast<uint2*>(out + col + g4 * 4) = make_uint2(pack_bf16(o.x * inv, o.y * inv), pack_bf16(o.z * inv, o.w * inv));
        }
    }
    __syncwarp();
    if (!softmax) cluster_arrive();
    cluster_wait();
}

// MANY: many more items than SMs.  A CTA then takes every gridDim.x-th one and keeps its tensor memory and barriers; the loads and
// the first S of the next item run under the tail of this one (layer-steps of 103 rows and 608 keys, us, one item per CTA | this:
// 64 requests 2678-2694 | 2659-2668, 40 requests 1756 | 1750; 60 rows and 396 keys, 30 requests 899 | 893; refresh of 90 rows
// over 192 keys, 64 requests, 2 layers 5841 | 5804; 28 heads, 64 requests of 105 rows 2790 | 2796; two runs differ by 0.3-0.8 %).
// With one item per CTA the same code was 1.7 us slower (103 rows over 1024 keys).
template <bool MANY>
__global__ void __launch_bounds__(AT_THREADS, 1)
attention_tc_kernel(const AttnTcArgs a, const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                    const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapKn,
                    const __grid_constant__ CUtensorMap mapVn) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint16_t row_max[4][128];  // [key quarter][row]: upper halves of fp32, rounded up
    __shared__ float row_sum[4][128];     // [key quarter][row]: shares of the denominator
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    if (base - smem_u32(smem_raw) > (uint32_t)AT_SLACK) {      // the tiles would not fit: report, touch nothing
        if (threadIdx.x == 0) atomicOr(a.status, kFlagWaitExpired);
        return;
    }
    const uint32_t sQ = base, sK0 = base + AT_TILE, sV0 = base + 3 * AT_TILE;
    const uint32_t bars = base + 5 * AT_TILE;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + 5 * AT_TILE + 192);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + 5 * AT_TILE + 200);
    // barriers: 0 q_full | 1,2 k_full | 3,4 k_empty | 5,6 v_full | 7,8 v_empty | 9,10 s_full | 11,12 unused |
    //           13,14 p_full | 15,16 pv_done (P V of the tile completed: O holds it, its S/P buffer is free)
    int* kept = reinterpret_cast<int*>(base_ptr + 5 * AT_TILE + 208);
    auto bar = [&](int i) { return bars + 8 * i; };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // key split: a cluster of C CTAs shares a query tile, each taking a contiguous part of the key tiles
    const int C = a.split, rank = C > 1 ? (int)cluster_ctarank() : 0;
    const int first = blockIdx.x / C, stride = gridDim.x;        // items: (query tile, head, request)
    const int n_cache_tiles = (a.ctx_len + 127) / 128;
    int2 visited = make_int2(0, n_cache_tiles);     // the cache's key tiles that hold keys
    // this CTA's key tiles: n_c of the cache from c0 on, then fresh ones from f0 on
    int qt, h, b, kvh, kb, live_q, c0, n_c, f0, n_tiles;
    auto set_item = [&](int item) {
        const int t = item / a.q_tiles;
        qt = item - t * a.q_tiles;
        b = t / a.n_heads;
        h = t - b * a.n_heads;
        kvh = h / (a.n_heads / a.n_kv_heads);
        kb = a.cache_shared ? 0 : b;                // one cache for the whole batch, or one per request
        const int all_tiles = n_cache_tiles + a.n_fresh_tiles;
        const int j0 = rank * all_tiles / C, j1 = (rank + 1) * all_tiles / C;
        c0 = max(j0, visited.x);
        n_c = max(min(j1, visited.y) - c0, 0);
        f0 = max(j0 - n_cache_tiles, 0);
        n_tiles = n_c + max(j1 - n_cache_tiles, 0) - f0;
        // 32-row quarters of the tile that hold rows: the softmax warps of the others have nothing to do (their
        // rows of S, P and O are never read), which matters when a decode pass brings 32 rows per request
        live_q = min(4, (a.n - qt * 128 + 31) / 32);
    };
    set_item(first);
    const int p_warps = MANY ? 16 : 4 * live_q;     // softmax warps that report a tile's P

    if (threadIdx.x == 0) {
        for (int i = 0; i <= 10; ++i) mbar_init(bar(i), 1);
        mbar_init(bar(13), p_warps); mbar_init(bar(14), p_warps);          // p_full
        mbar_init(bar(15), 1); mbar_init(bar(16), 1);      // pv_done
        *abort_flag = 0;
        kept[0] = INT_MAX; kept[1] = 0;
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
    const uint32_t tS0 = tmem_base, tO = tmem_base + 256;
    pdl_wait();
    pdl_launch_dependents();
    if (!MANY && C == 1 && a.pos_excl) {
        visited = kept_tiles(a, b, 1, kept);
        set_item(first);
    }

    const bool softmax = warp >= 2 && warp < 18 && (MANY || (warp & 3) < live_q);
    int J = 0;                                      // key tiles of the items before: ring stages and phases go on
    float m_use = -INFINITY, l = 0.f;               // softmax threads: exponent reference and denominator share of the row
    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        const uint64_t pol_q = policy_evict_first(), pol_kv = policy_evict_last();
        bool ok = true;
        for (int item = first; item < a.n_items && ok; item += stride, J += n_tiles) {
            if (MANY) set_item(item);
            // the last S of the item before has read Q
            if (J > 0 && !(ok = mbar_wait(bar(3 + ((J - 1) & 1)), ((J - 1) >> 1) & 1, abort_flag))) break;
            mbar_expect_tx(bar(0), AT_TILE);
            tma_load_3d(sQ, &mapQ, h * 128, qt * 128, b, bar(0), pol_q);
            tma_load_3d(sQ + AT_PANEL, &mapQ, h * 128 + 64, qt * 128, b, bar(0), pol_q);
            for (int j = 0; j < n_tiles && ok; ++j) {
                const int s = (J + j) & 1;
                const uint32_t par = (((J + j) >> 1) & 1) ^ 1;
                if (!(ok = mbar_wait(bar(3 + s), par, abort_flag))) break;
                const bool fresh = j >= n_c;
                const CUtensorMap* mk = fresh ? &mapKn : &mapK;
                const CUtensorMap* mv = fresh ? &mapVn : &mapV;
                const int r0 = (fresh ? f0 + j - n_c : c0 + j) * 128, bz = fresh ? b : kb;
                mbar_expect_tx(bar(1 + s), AT_TILE);
                tma_load_3d(sK0 + s * AT_TILE, mk, kvh * 128, r0, bz, bar(1 + s), pol_kv);
                tma_load_3d(sK0 + s * AT_TILE + AT_PANEL, mk, kvh * 128 + 64, r0, bz, bar(1 + s), pol_kv);
                if (!(ok = mbar_wait(bar(7 + s), par, abort_flag))) break;
                mbar_expect_tx(bar(5 + s), AT_TILE);
                tma_load_3d(sV0 + s * AT_TILE, mv, kvh * 128, r0, bz, bar(5 + s), pol_kv);
                tma_load_3d(sV0 + s * AT_TILE + AT_PANEL, mv, kvh * 128 + 64, r0, bz, bar(5 + s), pol_kv);
            }
            if (!MANY) break;
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer 1: S = Q K^T (M 128, N 128, both operands K-major) ----------------
        // The two products are issued by two threads of different warps: one thread doing both spends
        // more time in its four barrier waits and sixteen issues per tile than the tensor pipe needs
        // for the work.  Every tcgen05.commit tracks the issuing thread's own MMAs, and the cross
        // dependencies (P of tile j after S of tile j, S buffer reuse, O in tile order) all go through
        // mbarriers, so no ordering between the two threads is assumed.
        const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        bool ok = true;
        uint32_t q_par = 0;
        for (int item = first; item < a.n_items && ok; item += stride, J += n_tiles, q_par ^= 1) {
            if (MANY) set_item(item);
            ok = __all_sync(0xffffffffu, mbar_poll(bar(0), q_par, abort_flag));
            for (int j = 0; j < n_tiles && ok; ++j) {
                const int s = (J + j) & 1;
                const uint32_t par = ((J + j) >> 1) & 1;
                if (!(ok = __all_sync(0xffffffffu, mbar_poll(bar(1 + s), par, abort_flag)))) break;          // K of tile j landed
                // its S buffer also holds the P of tile j - 2: free once that tile's P V has completed
                if (J + j >= 2 && !(ok = __all_sync(0xffffffffu, mbar_poll(bar(15 + s), par ^ 1, abort_flag)))) break;
                tc_fence_after();
                const uint32_t k = sK0 + s * AT_TILE;
                if (elect_lane()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t da = smem_desc_sw128(sQ + (ks >> 2) * AT_PANEL) + (uint64_t)((ks & 3) * 2);
                        const uint64_t db = smem_desc_sw128(k + (ks >> 2) * AT_PANEL) + (uint64_t)((ks & 3) * 2);
                        tc_mma(tS0 + s * 128, da, db, idesc_s, ks > 0 ? 1u : 0u);
                    }
                    tc_commit(bar(9 + s));     // s_full
                    tc_commit(bar(3 + s));     // k_empty
                }
                __syncwarp();
            }
            if (!MANY) break;
        }
    } else if (warp == AT_THREADS / 32 - 1) {
        // ---------------- MMA issuer 2: O += P V (A = P K-major, B = V MN-major) ----------------
        const uint32_t idesc_o = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        // (the P of an item's first tile comes from threads that have read the O of the item before)
        bool ok = true;
        for (int item = first; item < a.n_items && ok; item += stride, J += n_tiles) {
            if (MANY) set_item(item);
            for (int j = 0; j < n_tiles && ok; ++j) {
                const int s = (J + j) & 1;
                const uint32_t par = ((J + j) >> 1) & 1;
                if (!(ok = __all_sync(0xffffffffu, mbar_poll(bar(13 + s), par, abort_flag)))) break;    // P of tile j written, O rescaled
                if (!(ok = __all_sync(0xffffffffu, mbar_poll(bar(5 + s), par, abort_flag)))) break;     // V of tile j landed
                tc_fence_after();
                const uint32_t v = sV0 + s * AT_TILE;
                if (elect_lane()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t db = smem_desc_mn_sw128(v + ks * 2048);
                        tc_mma_ta(tO, tS0 + s * 128 + ks * 8, db, idesc_o, (j > 0 || ks > 0) ? 1u : 0u);   // 16 keys = 8 columns of P
                    }
                    tc_commit(bar(15 + s));    // pv_done: O holds tiles 0..j, the S/P buffer is free
                    tc_commit(bar(7 + s));     // v_empty
                }
                __syncwarp();
            }
            if (!MANY) break;
        }
    } else if (softmax) {
        // ---------------- softmax: four threads per query row ----------------
        // Warp 2 + 4 c + q' (q = warp & 3 is its TMEM lane quarter) takes keys [32 c, 32 c + 32) of every
        // tile for the 32 rows of quarter q, and columns [32 c, 32 c + 32) of O.  Sixteen warps (four per
        // scheduler) keep the exponential, conversion and TMEM-load latencies of one warp hidden behind
        // the others.
        const int c4 = (warp - 2) >> 2;
        const int q = warp & 3;
        const int row = q * 32 + lane;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        const uint32_t col_off = (uint32_t)(c4 * 32);
        bool ok = true;
        for (int item = first; item < a.n_items; item += stride, J += n_tiles) {
            if (MANY) set_item(item);
            if (MANY && q >= live_q) {                  // no rows in this quarter: report its P as written
                for (int j = 0; j < n_tiles && ok; ++j) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar(9 + ((J + j) & 1)), ((J + j) >> 1) & 1, abort_flag));
                    if (ok && lane == 0) mbar_arrive(bar(13 + ((J + j) & 1)));
                }
                if (!ok) break;
                continue;
            }
            m_use = -INFINITY;
            l = 0.f;
            for (int j = 0; j < n_tiles; ++j) {
                const int s = (J + j) & 1;                // ring stage
                const uint32_t par = ((J + j) >> 1) & 1;
                // which of this thread's 32 keys count: the cache's positions up to the context end, minus those a
                // fresh row serves; of the fresh rows, those that serve their position
                uint32_t keep;
                if (j < n_c) {
                    const int w = (c0 + j) * 4 + c4, valid = a.ctx_len - w * 32;
                    keep = valid >= 32 ? 0xffffffffu : (valid <= 0 ? 0u : (1u << valid) - 1u);
                    if (a.pos_excl && w < a.excl_words) keep &= ~__ldg(a.pos_excl + (int64_t)b * a.excl_words + w);
                } else {
                    const int w = (f0 + j - n_c) * 4 + c4;
                    keep = w < a.keep_words ? __ldg(a.row_keep + (int64_t)b * a.keep_words + w) : 0u;
                }
                if (!softmax_tile(keep, j == 0, a.scale_log2e, tS0 + s * 128 + lane_off, tO + lane_off, c4, 1 + q, &row_max[0][row], 128,
                                  bar(13 + s), m_use, l, ok, [&] { return mbar_wait(bar(9 + s), par, abort_flag); },
                                  [&] { return mbar_wait(bar(15 + (s ^ 1)), ((J + j - 1) >> 1) & 1, abort_flag); }))
                    break;
            }
            // epilogue: O / l once the last P V has completed; the denominators of the four quarters add up
            if (ok && n_tiles > 0) ok = mbar_wait(bar(15 + ((J + n_tiles - 1) & 1)), ((J + n_tiles - 1) >> 1) & 1, abort_flag);
            row_sum[c4][row] = l;
            if (quarter_any(1 + q, !ok)) break;         // the four warps leave together
            l = (row_sum[0][row] + row_sum[1][row]) + (row_sum[2][row] + row_sum[3][row]);
            if (C == 1) {
                tc_fence_after();
                const int grow = qt * 128 + row;
                float v[32];
                tc_ld32(tO + lane_off + col_off, v);
                if (grow < a.n)
                    store_o32(static_cast<__nv_bfloat16*>(a.o) + (((int64_t)b * a.n + grow) * a.n_heads + h) * 128 + col_off, v, 1.f / l);
            }
            if (!MANY) break;
        }
    }
    if (C > 1) {
        const int c4 = (warp - 2) >> 2, row = (warp & 3) * 32 + lane, grow = qt * 128 + row;
        merge_parts(base, base_ptr, C, rank, softmax, n_tiles > 0, c4, row, tO + ((uint32_t)(warp & 3) << 21), m_use, l,
                    grow < a.n ? static_cast<__nv_bfloat16*>(a.o) + (((int64_t)b * a.n + grow) * a.n_heads + h) * 128 : nullptr);
    }
    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) {
            atomicOr(a.status, kFlagWaitExpired);
            for (int i = 0; i < 4096; ++i) __nanosleep(64);   // let copies already in flight land
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// ---- few rows per request over a shared cache ----------------------------------------------------
// Decode passes: the rows of `group` requests (four of at most 32 rows, or two of at most 64) share one 128-row query tile of one
// head, so that the shared cache's key tiles are read once per group.  First come those tiles, one step each, with the requests'
// own key masks.  Then come the requests' private rows, one round per 128 of them: every request's part of S (its 32-row quarter,
// or its two) is the product with its own key tile, written to its own lanes only (the instruction's disable-output-lane mask), and
// its part of O += P V likewise.  A round's softmax so works on as many logits as a shared tile's; with a step per (request, tile)
// three quarters of the softmax warps wrote zeros, and a step took as long as any.  16 requests of 32 rows, 32 heads, 2048 shared
// keys and 922 private rows, us a layer from the end of the launch before: 89 -> 75, with one barrier of a kind per shared step 72;
// 280 MB come from DRAM (42 us at the copy rate), 68 us for the launch alone.  A shared step is bound by the softmax chain (2700 cycles).
// What bounds a round (7300 cycles for 256 KB in one CTA's stamps: above the copy rate, part of it is there already) has not been separated:
// the loads, or the chain K, S, P, P V of a round.  Rounds and shared steps in turn, so that one's loads run under the other's
// arithmetic, were 9 us shorter, but another order of sums changes tokens that were near ties (2 of 512): not done.  Private
// tiles requested into L2 while the shared steps run: 7 to 17 us longer.  K and V rings of three stages.  96 registers, 8 bytes spilled.
constexpr int AG_STAGES = 3;
constexpr int AG_SMEM = (1 + 2 * AG_STAGES) * AT_TILE + 2048 + 512;    // Q, K, V, row exchange, barriers; the window has to start 1024-aligned

__global__ void __launch_bounds__(AT_THREADS, 1)
attention_group_kernel(const AttnTcArgs a, const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                       const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapKn,
                       const __grid_constant__ CUtensorMap mapVn) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if (base & 1023u) {                                        // the tiles would not be aligned: report, touch nothing
        if (threadIdx.x == 0) atomicOr(a.status, kFlagWaitExpired);
        return;
    }
    constexpr int kRows = (1 + 2 * AG_STAGES) * AT_TILE, kBars = kRows + 2048;
    const uint32_t sQ = base, sK0 = base + AT_TILE, sV0 = base + (1 + AG_STAGES) * AT_TILE, bars = base + kBars;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_raw + kBars + 352);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + kBars + 356);
    int* kept = reinterpret_cast<int*>(smem_raw + kBars + 360);
    // barriers: 0 q_full | by ring stage: 1.. k_full | 4.. k_empty | 7.. v_full | 10.. v_empty |
    //           by S buffer and, of a round, request: 13.. s_full | 21.. p_full | 29.. pv_done; of a shared step: 37.., 39.., 41..
    auto bar = [&](int i) { return bars + 8 * i; };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int C = a.split, rank = C > 1 ? (int)cluster_ctarank() : 0;
    const int G = a.group, qpr = 4 / G;                        // quarters per request
    const int item = blockIdx.x / C, h = item % a.n_heads, b0 = item / a.n_heads * G;
    const int n_req = min(G, a.batch - b0), live_q = n_req * qpr;
    const int kvh = h / (a.n_heads / a.n_kv_heads);

    if (warp == 0) {
        for (int i = lane; i < 43; i += 32) mbar_init(bar(i), i >= 21 && i < 29 ? 4 * qpr : i == 39 || i == 40 ? 4 * live_q : 1);
        if (lane == 0) {
            *abort_flag = 0;
            kept[0] = INT_MAX; kept[1] = 0;
        }
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
    const uint32_t tS0 = tmem_base, tO = tmem_base + 256;
    pdl_wait();
    pdl_launch_dependents();
    if (threadIdx.x == AT_THREADS - 32) {                      // (a warp that has nothing else to do yet)
        const uint64_t pol = policy_evict_first();
        mbar_expect_tx(bar(0), n_req * qpr * 8192);
        for (int r = 0; r < n_req; ++r) {                      // boxes of 32 qpr rows (rows past the request's read as zero)
            tma_load_3d(sQ + r * qpr * 4096, &mapQ, h * 128, 0, b0 + r, bar(0), pol);
            tma_load_3d(sQ + AT_PANEL + r * qpr * 4096, &mapQ, h * 128 + 64, 0, b0 + r, bar(0), pol);
        }
    }
    __syncwarp();
    const int n_cache = (a.ctx_len + 127) / 128;
    const int2 cache = C == 1 ? kept_tiles(a, b0, n_req, kept) : make_int2(0, n_cache);

    // This CTA's part: the key tiles, the cache's and then request by request the private ones, are cut into C ranges; of those that
    // hold keys n_s shared ones from t0 on, then n_own(r) private ones of request r from f_own(r) on, one in each round.
    const int n_all = n_cache + a.n_fresh_tiles * n_req;
    const int j0 = rank * n_all / C, j1 = (rank + 1) * n_all / C;
    const int t0 = max(j0, cache.x), n_s = max(min(j1, cache.y) - t0, 0);
    auto f_own = [&](int r) { return min(max(j0 - n_cache - r * a.n_fresh_tiles, 0), a.n_fresh_tiles); };
    auto n_own = [&](int r) { return min(max(j1 - n_cache - r * a.n_fresh_tiles, 0), a.n_fresh_tiles) - f_own(r); };
    int n_steps = 0;
    for (int r = 0; r < n_req; ++r) n_steps = max(n_steps, n_own(r));
    n_steps += n_s;
    // Barrier and phase of step i, request r: s_full, p_full, pv_done.  A shared step is one product for all requests and has one
    // barrier of each kind: with every request's own ones the two issuing warps waited and committed up to four times a step (32
    // heads, 32 rows a request: 6 requests over 4096 shared keys 68.5 -> 65.0 us, 16 over 2048 70 -> 66).
    auto s_full = [&](int i, int r) { return bar(i < n_s ? 37 + (i & 1) : 13 + (i & 1) * 4 + r); };
    auto p_full = [&](int i, int r) { return bar(i < n_s ? 39 + (i & 1) : 21 + (i & 1) * 4 + r); };
    auto pv_done = [&](int i, int r) { return bar(i < n_s ? 41 + (i & 1) : 29 + (i & 1) * 4 + r); };
    auto phase = [&](int i) { return (uint32_t)((i < n_s ? i : i - n_s) >> 1) & 1u; };

    const bool softmax = warp >= 2 && warp < 18 && (warp & 3) < live_q;
    const int n_mine = n_s + (softmax ? n_own((warp & 3) / qpr) : 0);      // steps of this warp's request
    float m_use = -INFINITY, l = 0.f;
    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer: K and V rings each as far ahead as they go ----------------
        const uint64_t pol_shared = policy_evict_last(), pol_own = policy_evict_first();
        int ki = 0, vi = 0, kr = 0, vr = 0, ks = 0, vs = 0;    // where each ring is: step, request of a round, stage, phase
        uint32_t kp = 1, vp = 1;
        auto settle = [&](int& i, int& r) {                    // on to the next request that has a tile in the round
            while (i >= n_s && i < n_steps && (r == n_req || i - n_s >= n_own(r)))
                if (++r >= n_req) { r = 0; ++i; }
        };
        auto load = [&](int& i, int& r, uint32_t dst, uint32_t full, const CUtensorMap* shared_map, const CUtensorMap* own_map) {
            const bool own = i >= n_s;
            const CUtensorMap* m = own ? own_map : shared_map;
            const int r0 = (own ? f_own(r) + i - n_s : t0 + i) * 128, bz = own ? b0 + r : 0;
            const uint64_t pol = own ? pol_own : pol_shared;
            mbar_expect_tx(full, AT_TILE);
            tma_load_3d(dst, m, kvh * 128, r0, bz, full, pol);
            tma_load_3d(dst + AT_PANEL, m, kvh * 128 + 64, r0, bz, full, pol);
            if (own) ++r;
            else ++i;
            settle(i, r);
        };
        settle(ki, kr);
        settle(vi, vr);
        for (uint32_t idle = 0; ki < n_steps || vi < n_steps;) {
            bool moved = false;
            if (ki < n_steps && mbar_test(bar(4 + ks), kp)) {
                load(ki, kr, sK0 + ks * AT_TILE, bar(1 + ks), &mapK, &mapKn);
                if (++ks == AG_STAGES) { ks = 0; kp ^= 1; }
                moved = true;
            }
            if (vi < n_steps && mbar_test(bar(10 + vs), vp)) {
                load(vi, vr, sV0 + vs * AT_TILE, bar(7 + vs), &mapV, &mapVn);
                if (++vs == AG_STAGES) { vs = 0; vp ^= 1; }
                moved = true;
            }
            if (moved) idle = 0;
            else if (++idle >= TC_WAIT_LIMIT << 4) *abort_flag = 1;
            if ((idle & 1023u) == 1023u && *abort_flag) break;
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer 1: S = Q K^T ----------------
        const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        auto wait = [&](uint32_t b, uint32_t parity) { return __all_sync(0xffffffffu, mbar_poll(b, parity, abort_flag)); };
        bool ok = wait(bar(0), 0);
        int ks = 0;
        uint32_t kp = 0;
        for (int i = 0; i < n_steps && ok; ++i) {
            const bool own = i >= n_s;
            const int parts = own ? n_req : 1;                 // a product per request, or one for all of them
            for (int r = 0; r < parts && ok; ++r) {
                if (own && i - n_s >= n_own(r)) continue;
                // the S buffer also holds the P of step i - 2: free once that step's P V has completed
                if (i >= 2) ok = wait(pv_done(i - 2, r), phase(i - 2));
                if (!ok || !(ok = wait(bar(1 + ks), kp))) break;                  // K landed
                tc_fence_after();
                const uint32_t k = sK0 + ks * AT_TILE;
                const uint32_t lanes = own ? ((1u << qpr) - 1u) << (r * qpr) : 15u;
                if (elect_lane()) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const uint64_t da = smem_desc_sw128(sQ + (e >> 2) * AT_PANEL) + (uint64_t)((e & 3) * 2);
                        const uint64_t db = smem_desc_sw128(k + (e >> 2) * AT_PANEL) + (uint64_t)((e & 3) * 2);
                        tc_mma_lanes(tS0 + (i & 1) * 128, da, db, idesc_s, e > 0 ? 1u : 0u, lanes);
                    }
                    tc_commit(s_full(i, r));
                    tc_commit(bar(4 + ks));            // k_empty
                }
                __syncwarp();
                if (++ks == AG_STAGES) { ks = 0; kp ^= 1; }
            }
        }
    } else if (warp == AT_THREADS / 32 - 1) {
        // ---------------- MMA issuer 2: O += P V ----------------
        const uint32_t idesc_o = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        auto wait = [&](uint32_t b, uint32_t parity) { return __all_sync(0xffffffffu, mbar_poll(b, parity, abort_flag)); };
        bool ok = true;
        int vs = 0;
        uint32_t vp = 0;
        for (int i = 0; i < n_steps && ok; ++i) {
            const bool own = i >= n_s;
            const int parts = own ? n_req : 1;
            for (int r = 0; r < parts && ok; ++r) {
                if (own && i - n_s >= n_own(r)) continue;
                if (!(ok = wait(p_full(i, r), phase(i))) || !(ok = wait(bar(7 + vs), vp))) break;      // P written, O rescaled; V landed
                tc_fence_after();
                const uint32_t v = sV0 + vs * AT_TILE;
                const uint32_t lanes = own ? ((1u << qpr) - 1u) << (r * qpr) : 15u;
                if (elect_lane()) {
#pragma unroll
                    for (int e = 0; e < 8; ++e)                    // 16 keys = 8 columns of P
                        tc_mma_ta_lanes(tO, tS0 + (i & 1) * 128 + e * 8, smem_desc_mn_sw128(v + e * 2048), idesc_o,
                                        (i > 0 || e > 0) ? 1u : 0u, lanes);
                    tc_commit(pv_done(i, r));
                    tc_commit(bar(10 + vs));           // v_empty
                }
                __syncwarp();
                if (++vs == AG_STAGES) { vs = 0; vp ^= 1; }
            }
        }
    } else if (softmax) {
        // ---------------- softmax: four threads per query row, as in the one-tile kernel ----------------
        const int c4 = (warp - 2) >> 2, q = warp & 3, r = q / qpr;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        // per quarter: the exchange of maxima [4][32], and of denominators [4][32] when the last tile is done
        uint16_t* row_max = reinterpret_cast<uint16_t*>(smem_raw + kRows + q * 512) + lane;
        float* row_sum = reinterpret_cast<float*>(smem_raw + kRows + q * 512) + lane;
        bool ok = true;
        const uint32_t* excl = a.pos_excl + (int64_t)(b0 + r) * a.excl_words;
        const uint32_t* serves = a.row_keep + (int64_t)(b0 + r) * a.keep_words;
        int w = (n_s > 0 ? t0 : f_own(r)) * 4 + c4;            // this thread's word of the step's key masks
        auto keys = [&](bool own) {                            // which of its 32 keys count
            if (own) return w < a.keep_words ? __ldg(serves + w) : 0u;
            const int valid = a.ctx_len - w * 32;
            const uint32_t in = valid >= 32 ? ~0u : (valid <= 0 ? 0u : (1u << valid) - 1u);
            return w < a.excl_words ? in & ~__ldg(excl + w) : in;
        };
        uint32_t next = n_mine > 0 ? keys(n_s == 0) : 0u;      // asked for a step ahead
        for (int i = 0; i < n_mine; ++i) {
            const uint32_t keep = next;
            w = i + 1 == n_s ? f_own(r) * 4 + c4 : w + 4;
            if (i + 1 < n_mine) next = keys(i + 1 >= n_s);
            if (!softmax_tile(keep, i == 0, a.scale_log2e, tS0 + (i & 1) * 128 + lane_off, tO + lane_off, c4, 1 + q, row_max, 32,
                              p_full(i, r), m_use, l, ok, [&] { return mbar_wait(s_full(i, r), phase(i), abort_flag); },
                              [&] { return mbar_wait(pv_done(i - 1, r), phase(i - 1), abort_flag); }))
                break;
        }
        // O / l once the last P V has completed (every thread of the row has read the maxima by then)
        if (ok && n_mine > 0) ok = mbar_wait(pv_done(n_mine - 1, r), phase(n_mine - 1), abort_flag);
        row_sum[c4 * 32] = l;
        if (!quarter_any(1 + q, !ok)) {
            l = (row_sum[0] + row_sum[32]) + (row_sum[64] + row_sum[96]);
            if (C == 1) {
                tc_fence_after();
                const int grow = (q - r * qpr) * 32 + lane;
                float v[32];
                tc_ld32(tO + lane_off + c4 * 32, v);
                if (grow < a.n)
                    store_o32(static_cast<__nv_bfloat16*>(a.o) + (((int64_t)(b0 + r) * a.n + grow) * a.n_heads + h) * 128 + c4 * 32, v, 1.f / l);
            }
        }
    }
    if (C > 1) {
        __syncwarp();
        __syncthreads();              // a request without tiles of its own here is done before the others' products have read K
        const int q = warp & 3, r = q / qpr, grow = (q - r * qpr) * 32 + lane;
        merge_parts(base, smem_raw, C, rank, softmax, n_mine > 0, (warp - 2) >> 2, q * 32 + lane, tO + ((uint32_t)q << 21), m_use, l,
                    r < n_req && grow < a.n ? static_cast<__nv_bfloat16*>(a.o) + (((int64_t)(b0 + r) * a.n + grow) * a.n_heads + h) * 128
                                            : nullptr);
    }
    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) {
            atomicOr(a.status, kFlagWaitExpired);
            for (int i = 0; i < 4096; ++i) __nanosleep(64);   // let copies already in flight land
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// ---- two query tiles per CTA ------------------------------------------------------------------
// 256 query rows of one head share every K/V tile that lands in shared memory.  Each 128-row query tile
// has its own S buffer, O accumulator and softmax warps (one thread per row: the row maximum needs no
// exchange).  The softmax works through a tile's 128 keys in two halves of 64 (so that a row's values
// fit in registers without spilling) and writes each half's P over the low columns of the S buffer; one
// thread issues everything: the P V of a half as soon as that half's P is there, and after the second
// half the tile's next S into the same buffer (the tensor pipe executes one thread's instructions in
// order).  While one query tile's softmax runs, the tensor pipe works on the other's.  Measured and not
// kept: S as two 64-key products into two buffers per query tile (a 128 x 64 x 16 product holds the
// issuing thread as long as a 128 x 128 x 16 one: 74 against 66 cycles), and one issuing thread per query
// tile (their interleaved instructions ran slower than one thread's fixed order).
//
// The exponent reference of a row only moves when a half's maximum exceeds it by more than 2^8 (then O
// and the denominator are rescaled), so the common path is: x = s * scale - reference (two per FFMA2),
// maximum, exp2 (a quarter of them on the FMA pipe), bf16 pack, store to tensor memory.
constexpr int AT2_THREADS = 320;                 // warp 0: TMA, warp 1: MMA issuer, warps 2-5 / 6-9: softmax of query tile 0 / 1
constexpr int AT2_SMEM = 6 * AT_TILE + AT_SLACK + 256 + 2048;   // Q x2, K x2, V x2, barriers, score tables

__device__ __forceinline__ void tc_ld32_nowait(uint32_t taddr, float (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
          "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]),
          "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]), "=f"(v[24]),
          "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
        : "r"(taddr)
        : "memory");
}
// The loads above are complete after this; the values pass through it so that no use can move ahead of it.
__device__ __forceinline__ void tc_wait_ld32(float (&v)[32]) {
    asm volatile(
        "tcgen05.wait::ld.sync.aligned;"
        : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]),
          "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]), "+f"(v[16]),
          "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]), "+f"(v[23]), "+f"(v[24]),
          "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]), "+f"(v[30]), "+f"(v[31])
        :
        : "memory");
}
__device__ __forceinline__ void tc_st32u(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
          "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]),
          "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]),
          "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

__global__ void __launch_bounds__(AT2_THREADS, 1)
attention_tc2q_kernel(const AttnTcArgs a, const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                      const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapKn,
                      const __grid_constant__ CUtensorMap mapVn) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    if (base - smem_u32(smem_raw) > (uint32_t)AT_SLACK) {      // the tiles would not fit: report, touch nothing
        if (threadIdx.x == 0) atomicOr(a.status, kFlagWaitExpired);
        return;
    }
    const uint32_t sQ = base, sK0 = base + 2 * AT_TILE, sV0 = base + 4 * AT_TILE;
    const uint32_t bars = base + 6 * AT_TILE;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + 6 * AT_TILE + 192);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + 6 * AT_TILE + 200);
    // barriers: 0 q_full | 1,2 k_full | 3,4 k_empty | 5,6 v_full | 7,8 v_empty | 9 + t: s_full |
    //           11 + 2 t + hb: p_full | 15 + 2 t + hb: pv_done   (query tile t, key half hb)
    auto bar = [&](int i) { return bars + 8 * i; };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int qt = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int kvh = h / (a.n_heads / a.n_kv_heads);
    int* kept = reinterpret_cast<int*>(base_ptr + 6 * AT_TILE + 208);
    const int kb = a.cache_shared ? 0 : b;
    const int n_sets = (qt * 256 + 128 < a.n) ? 2 : 1;      // the last CTA of an odd tile count has one tile
    float2* s_tab = reinterpret_cast<float2*>(base_ptr + 6 * AT_TILE + 256);     // [2 query tiles][128 rows] (reference, weight)

    if (threadIdx.x == 0) {
        for (int i = 0; i <= 10; ++i) mbar_init(bar(i), 1);
        for (int i = 11; i <= 14; ++i)                         // p_full: the softmax warps of the query tile that have rows
            mbar_init(bar(i), max(1, min(4, (a.n - qt * 256 - (i >= 13 ? 128 : 0) + 31) / 32)));
        for (int i = 15; i <= 18; ++i) mbar_init(bar(i), 1);
        mbar_init(bar(19), 4); mbar_init(bar(20), 4);          // score sweep: the four warps of a query tile are done with D
        *abort_flag = 0;
        kept[0] = INT_MAX; kept[1] = 0;
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
    // columns: S of query tile 0 | S of query tile 1 | O of query tile 0 | O of query tile 1, 128 each
    pdl_wait();
    pdl_launch_dependents();
    const int2 cache = kept_tiles(a, b, 1, kept);
    const int c_lo = cache.x, n_cache_tiles = cache.y - cache.x, n_tiles = n_cache_tiles + a.n_fresh_tiles;
    // score sweep (Eq. 4-5 from this attention's logits): only CTAs whose 256 query rows hold a flagged row walk the
    // affix key tiles [sw0, sw0 + n_sw) a second time
    int n_sw = 0, sw0 = 0;
    if (a.score_rowmask && a.affix_len > 0) {
        uint32_t any = 0u;
        for (int w = qt * 8; w < min(qt * 8 + 8, a.rm_words); ++w) any |= __ldg(a.score_rowmask + (int64_t)b * a.rm_words + w);
        if (any) { sw0 = a.affix_start >> 7; n_sw = ((a.affix_start + a.affix_len - 1) >> 7) - sw0 + 1; }
    }

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        const uint64_t pol_q = policy_evict_first(), pol_kv = policy_evict_last();
        mbar_expect_tx(bar(0), n_sets * AT_TILE);
        for (int t = 0; t < n_sets; ++t) {
            tma_load_3d(sQ + t * AT_TILE, &mapQ, h * 128, qt * 256 + t * 128, b, bar(0), pol_q);
            tma_load_3d(sQ + t * AT_TILE + AT_PANEL, &mapQ, h * 128 + 64, qt * 256 + t * 128, b, bar(0), pol_q);
        }
        // K/V tiles a few iterations ahead are requested into L2, so that the loads into the two-stage rings
        // (issued one iteration before use) do not wait on HBM
        auto prefetch_tile = [&](int j) {
            if (j >= n_tiles) return;
            const bool fresh = j >= n_cache_tiles;
            const int r0 = (fresh ? j - n_cache_tiles : c_lo + j) * 128, bz = fresh ? b : kb;
            tma_prefetch_3d(fresh ? &mapKn : &mapK, kvh * 128, r0, bz);
            tma_prefetch_3d(fresh ? &mapKn : &mapK, kvh * 128 + 64, r0, bz);
            tma_prefetch_3d(fresh ? &mapVn : &mapV, kvh * 128, r0, bz);
            tma_prefetch_3d(fresh ? &mapVn : &mapV, kvh * 128 + 64, r0, bz);
        };
        for (int j = 2; j < 2 + a.kv_prefetch; ++j) prefetch_tile(j);
        bool ok = true;
        for (int j = 0; j < n_tiles && ok; ++j) {
            const int s = j & 1;
            const uint32_t par = ((j >> 1) & 1) ^ 1;
            if (a.kv_prefetch) prefetch_tile(j + 2 + a.kv_prefetch);
            if (!(ok = mbar_wait(bar(3 + s), par, abort_flag))) break;
            const bool fresh = j >= n_cache_tiles;
            const CUtensorMap* mk = fresh ? &mapKn : &mapK;
            const CUtensorMap* mv = fresh ? &mapVn : &mapV;
            const int r0 = (fresh ? j - n_cache_tiles : c_lo + j) * 128, bz = fresh ? b : kb;
            mbar_expect_tx(bar(1 + s), AT_TILE);
            tma_load_3d(sK0 + s * AT_TILE, mk, kvh * 128, r0, bz, bar(1 + s), pol_kv);
            tma_load_3d(sK0 + s * AT_TILE + AT_PANEL, mk, kvh * 128 + 64, r0, bz, bar(1 + s), pol_kv);
            if (!(ok = mbar_wait(bar(7 + s), par, abort_flag))) break;
            mbar_expect_tx(bar(5 + s), AT_TILE);
            tma_load_3d(sV0 + s * AT_TILE, mv, kvh * 128, r0, bz, bar(5 + s), pol_kv);
            tma_load_3d(sV0 + s * AT_TILE + AT_PANEL, mv, kvh * 128 + 64, r0, bz, bar(5 + s), pol_kv);
        }
        for (int js = 0; js < n_sw && ok; ++js) {            // the affix key tiles once more (keys only)
            const int jj = n_tiles + js, s = jj & 1;
            if (!(ok = mbar_wait(bar(3 + s), ((jj >> 1) & 1) ^ 1, abort_flag))) break;
            mbar_expect_tx(bar(1 + s), AT_TILE);
            tma_load_3d(sK0 + s * AT_TILE, &mapK, kvh * 128, (sw0 + js) * 128, kb, bar(1 + s), pol_kv);
            tma_load_3d(sK0 + s * AT_TILE + AT_PANEL, &mapK, kvh * 128 + 64, (sw0 + js) * 128, kb, bar(1 + s), pol_kv);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the whole warp runs the loop, one lane issues ----------------
        // (with one lane in the loop, refresh of 14 752 rows 12 579 -> 12 524 us here, layer-step of 103 rows 144.0 -> 143.8 us
        // in the one-tile kernel)
        const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t idesc_o = idesc_s | (1u << 16);       // B = V is MN-major
        auto wait = [&](int i, uint32_t parity) { return __all_sync(0xffffffffu, mbar_poll(bar(i), parity, abort_flag)); };
        auto issue_s = [&](int t, int j) {                   // S_t = Q_t K_j^T, then s_full of query tile t
            const uint32_t k = sK0 + (j & 1) * AT_TILE;
            if (!elect_lane()) return;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                const uint64_t da = smem_desc_sw128(sQ + t * AT_TILE + (ks >> 2) * AT_PANEL) + (uint64_t)((ks & 3) * 2);
                const uint64_t db = smem_desc_sw128(k + (ks >> 2) * AT_PANEL) + (uint64_t)((ks & 3) * 2);
                tc_mma(tmem_base + t * 128, da, db, idesc_s, ks > 0 ? 1u : 0u);
            }
            tc_commit(bar(9 + t));
        };
        bool ok = wait(0, 0);
        if (ok && n_tiles > 0 && (ok = wait(1, 0))) {
            tc_fence_after();
            for (int t = 0; t < n_sets; ++t) issue_s(t, 0);
            if (elect_lane()) tc_commit(bar(3));             // k_empty of stage 0
            __syncwarp();
        }
        for (int j = 0; j < n_tiles && ok; ++j) {
            const int s = j & 1;
            const bool more = j + 1 < n_tiles;
            if (!(ok = wait(5 + s, (j >> 1) & 1))) break;                       // V of tile j landed
            if (more && !(ok = wait(1 + (s ^ 1), ((j + 1) >> 1) & 1))) break;   // K of tile j + 1 landed
            const uint32_t v = sV0 + s * AT_TILE;
            for (int t = 0; t < n_sets && ok; ++t) {
                for (int hb = 0; hb < 2 && ok; ++hb) {
                    if (!(ok = wait(11 + 2 * t + hb, j & 1))) break;  // P of this half written, O rescaled
                    tc_fence_after();
                    if (elect_lane()) {
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4) {
                            const int ks = hb * 4 + k4;          // 16 keys = 8 columns of P
                            tc_mma_ta(tmem_base + 256 + t * 128, tmem_base + t * 128 + ks * 8, smem_desc_mn_sw128(v + ks * 2048), idesc_o,
                                      (j > 0 || ks > 0) ? 1u : 0u);
                        }
                        tc_commit(bar(15 + 2 * t + hb));         // pv_done: O holds everything up to this half
                    }
                    __syncwarp();
                }
                if (ok && more) issue_s(t, j + 1);           // overwrites P: executes after the P V just issued
                __syncwarp();
            }
            if (elect_lane()) {
                tc_commit(bar(7 + s));                           // v_empty
                if (more) tc_commit(bar(3 + (s ^ 1)));           // k_empty of tile j + 1
            }
            __syncwarp();
        }
        // score sweep: D_t = K Q_t^T into the S buffer of query tile t (its last P V was issued above by this thread, and
        // the tensor pipe keeps one thread's instructions in order)
        for (int js = 0; js < n_sw && ok; ++js) {
            const int jj = n_tiles + js, s = jj & 1;
            if (!(ok = wait(1 + s, (jj >> 1) & 1))) break;
            const uint32_t k = sK0 + s * AT_TILE;
            for (int t = 0; t < n_sets && ok; ++t) {
                if (js > 0 && !(ok = wait(19 + t, (js - 1) & 1))) break;
                tc_fence_after();
                if (elect_lane()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t da = smem_desc_sw128(k + (ks >> 2) * AT_PANEL) + (uint64_t)((ks & 3) * 2);
                        const uint64_t db = smem_desc_sw128(sQ + t * AT_TILE + (ks >> 2) * AT_PANEL) + (uint64_t)((ks & 3) * 2);
                        tc_mma(tmem_base + t * 128, da, db, idesc_s, ks > 0 ? 1u : 0u);
                    }
                    tc_commit(bar(9 + t));
                }
                __syncwarp();
            }
            if (ok && elect_lane()) tc_commit(bar(3 + s));   // k_empty
            __syncwarp();
        }
    } else if (warp >= 2 && warp < 2 + 4 * n_sets) {
      const int t = (warp - 2) >> 2;
      const int q = warp & 3;                              // the warp's TMEM lane quarter
      const int row = q * 32 + lane;
      const uint32_t lane_off = (uint32_t)(q * 32) << 16;
      const uint32_t tS = tmem_base + t * 128 + lane_off, tO = tmem_base + 256 + t * 128 + lane_off;
      const bool has_rows = q * 32 < a.n - qt * 256 - t * 128;
      // Eq. 4 normalises over the affix keys: the denominator restricted to them is kept next to the full one
      const bool want_lf = n_sw > 0 && !a.score_norm_full;
      float m_use = -INFINITY, l = 0.f, lf = 0.f;
      bool ok = true;
      if (has_rows) {
        // ---------------- softmax: one thread per query row ----------------
        const float2 sc2 = make_float2(a.scale_log2e, a.scale_log2e);
        // The keys that count are worked out a tile at a time, before the wait for its S, and not at all for tiles that lie whole
        // inside the context and inside or outside the affix span: worked out per half they took some 400 cycles between the first
        // half's P and the second half's logits, on the chain of every tile.  With the issuing warp's waits as polls: 14 752 rows
        // over 2560 keys 790 -> 768 us alone, 1095 -> 1063 back to back under the power cap.  Bound by that chain still (of 5000
        // cycles per key tile and two query tiles 1900 are issue, 2200 tensor work), not by a unit.
        uint32_t keep4[4] = {~0u, ~0u, ~0u, ~0u}, aff4[4] = {0u, 0u, 0u, 0u};
        const int aff0 = a.affix_start, aff1 = a.affix_start + a.affix_len;
        for (int i = 0; i < 2 * n_tiles && ok; ++i) {
            const int hb = i & 1, j = i >> 1;
            if (hb == 0) {
                const int k0 = (c_lo + j) * 128;                  // (of a cache tile)
                const bool in = !want_lf || (k0 >= aff0 && k0 + 128 <= aff1), out = !want_lf || k0 >= aff1 || k0 + 128 <= aff0;
                if (!a.pos_excl && k0 + 128 <= a.ctx_len && (in || out)) {
#pragma unroll
                    for (int w = 0; w < 4; ++w) { keep4[w] = ~0u; aff4[w] = want_lf && in ? ~0u : 0u; }
                } else {
                    // which of the tile's keys count: the cache's positions up to the context end, minus those a fresh row
                    // serves; of the fresh rows, those that serve their position
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        aff4[w] = 0u;
                        if (j < n_cache_tiles) {
                            const int valid = a.ctx_len - k0 - w * 32;
                            keep4[w] = valid >= 32 ? ~0u : (valid <= 0 ? 0u : (1u << valid) - 1u);
                            if (a.pos_excl && (k0 >> 5) + w < a.excl_words) keep4[w] &= ~__ldg(a.pos_excl + (int64_t)b * a.excl_words + (k0 >> 5) + w);
                            // of those keys, the ones inside the affix span
                            const int lo = max(aff0 - k0 - w * 32, 0), hi = min(aff1 - k0 - w * 32, 32);
                            if (want_lf && hi > lo) aff4[w] = (hi - lo >= 32 ? ~0u : ((1u << (hi - lo)) - 1u) << lo);
                        } else {
                            const int fw = (j - n_cache_tiles) * 4 + w;
                            keep4[w] = fw < a.keep_words ? __ldg(a.row_keep + (int64_t)b * a.keep_words + fw) : 0u;
                        }
                    }
                }
            }
            const uint32_t keep[2] = {hb ? keep4[2] : keep4[0], hb ? keep4[3] : keep4[1]};
            const uint32_t aff[2] = {hb ? aff4[2] : aff4[0], hb ? aff4[3] : aff4[1]};
            const bool aff_all = (aff[0] & aff[1]) == ~0u, aff_none = (aff[0] | aff[1]) == 0u;
            const bool all = (keep[0] & keep[1]) == ~0u && (aff_all || aff_none);
            // warp-uniform: the tensor-memory accesses below are collective
            if (hb == 0) {
                if (!(ok = __all_sync(0xffffffffu, mbar_spin(bar(9 + t), j & 1, abort_flag)))) break;
                tc_fence_after();
            }
            float sv[2][32];
            tc_ld32_nowait(tS + hb * 64, sv[0]);
            tc_ld32_nowait(tS + hb * 64 + 32, sv[1]);
            tc_wait_ld32(sv[0]);
            tc_wait_ld32(sv[1]);
            // x = s * scale - reference, in place; the reference is 0 until a half with a key that counts
            const bool first = m_use == -INFINITY;
            const float m_ref = first ? 0.f : m_use;
            const float2 mr2 = make_float2(-m_ref, -m_ref);
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float2 r = __ffma2_rn(make_float2(sv[c][2 * e], sv[c][2 * e + 1]), sc2, mr2);
                    sv[c][2 * e] = r.x;
                    sv[c][2 * e + 1] = r.y;
                }
            // masked keys as -inf: their P is 0
            if (!all) {
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int e = 0; e < 32; ++e) sv[c][e] = ((keep[c] >> e) & 1u) ? sv[c][e] : -INFINITY;
            }
            float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int e = 0; e < 32; e += 2) m4[(e >> 1) & 3] = fmaxf(fmaxf(m4[(e >> 1) & 3], sv[c][e]), sv[c][e + 1]);
            const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
            const bool raise = mx > kRescaleGap || (first && mx > -INFINITY);
            if (__any_sync(0xffffffffu, raise)) {
                const float f = raise ? (first ? 0.f : fast_exp2(-mx)) : 1.f;
                if (i > 0) {
                    // O may only be touched once the P V of half i - 1 (and with it every earlier one) has completed
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(bar(15 + 2 * t + ((i - 1) & 1)), ((i - 1) >> 1) & 1, abort_flag)))) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        float v[32];
                        tc_ld32(tO + c * 32, v);
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] *= f;
                        tc_st32(tO + c * 32, v);
                    }
                    tc_wait_st();
                }
                l *= f;
                lf *= f;
                if (raise) {
                    m_use = m_ref + mx;
#pragma unroll
                    for (int c = 0; c < 2; ++c)
#pragma unroll
                        for (int e = 0; e < 32; ++e) sv[c][e] -= mx;
                }
            }
            // P as packed bf16: the half's 64 keys go to columns 32 hb .. 32 hb + 31 of the S buffer, over S values of
            // keys below 64 that this thread read in the first half
            float2 l2a = make_float2(0.f, 0.f), l2b = make_float2(0.f, 0.f), lf2 = make_float2(0.f, 0.f);
            uint32_t pk[32];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (all) {
#pragma unroll
                    for (int e = 0; e < 32; e += 4) {
                        const float2 pa = make_float2(fast_exp2(sv[c][e]), fast_exp2(sv[c][e + 1]));
                        const float2 pb = make_float2(fast_exp2(sv[c][e + 2]), poly_exp2(sv[c][e + 3]));
                        l2a = __fadd2_rn(l2a, pa);
                        l2b = __fadd2_rn(l2b, pb);
                        pk[c * 16 + (e >> 1)] = pack_bf16(pa.x, pa.y);
                        pk[c * 16 + (e >> 1) + 1] = pack_bf16(pb.x, pb.y);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        const float p0 = fast_exp2(sv[c][e]), p1 = fast_exp2(sv[c][e + 1]);
                        l2a = __fadd2_rn(l2a, make_float2(p0, p1));
                        lf2 = __fadd2_rn(lf2, make_float2(((aff[c] >> e) & 1u) ? p0 : 0.f, ((aff[c] >> (e + 1)) & 1u) ? p1 : 0.f));
                        pk[c * 16 + (e >> 1)] = pack_bf16(p0, p1);
                    }
                }
            }
            tc_st32u(tS + hb * 32, pk);
            tc_wait_st();
            const float half_sum = (l2a.x + l2a.y) + (l2b.x + l2b.y);
            l += half_sum;
            lf += all ? (aff_all ? half_sum : 0.f) : (lf2.x + lf2.y);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(11 + 2 * t + hb));   // p_full
        }
        // epilogue: O / l once the last P V has completed
        if (ok && n_tiles > 0) ok = __all_sync(0xffffffffu, mbar_wait(bar(15 + 2 * t + 1), (n_tiles - 1) & 1, abort_flag));
        if (ok) {
            tc_fence_after();
            const int grow = qt * 256 + t * 128 + row;
            const float inv = 1.f / l;
            __nv_bfloat16* out = static_cast<__nv_bfloat16*>(a.o) + (((int64_t)b * a.n + grow) * a.n_heads + h) * 128;
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                float v[32];
                tc_ld32(tO + c * 32, v);
                if (grow < a.n) {
#pragma unroll
                    for (int k8 = 0; k8 < 4; ++k8) {
                        const float* pv = v + k8 * 8;
                        *reinterpret_cast<uint4*>(out + c * 32 + k8 * 8) =
                            make_uint4(pack_bf16(pv[0] * inv, pv[1] * inv), pack_bf16(pv[2] * inv, pv[3] * inv),
                                       pack_bf16(pv[4] * inv, pv[5] * inv), pack_bf16(pv[6] * inv, pv[7] * inv));
                    }
                }
            }
        }
      }
      if (n_sw > 0) {
        // ---------------- score sweep: thread = key, columns = the query rows of tile t ----------------
        // every row's (reference, weight): weight = 1 / (its denominator over the affix keys) for a flagged row, else 0
        {
            const int grow = qt * 256 + t * 128 + row;
            float w = 0.f;
            const float den = a.score_norm_full ? l : lf;
            if (has_rows && ok && grow < a.n && den > 0.f &&
                ((__ldg(a.score_rowmask + (int64_t)b * a.rm_words + (grow >> 5)) >> (grow & 31)) & 1u))
                w = 1.f / den;
            s_tab[t * 128 + row] = make_float2(has_rows && m_use > -INFINITY ? m_use : 0.f, w);
        }
        asm volatile("bar.sync %0, 128;" ::"r"(1 + t) : "memory");     // the four warps of query tile t
        uint32_t nz = 0u;                                              // 32-row column chunks that hold a flagged row
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (__any_sync(0xffffffffu, s_tab[t * 128 + c * 32 + lane].y != 0.f)) nz |= 1u << c;
        for (int js = 0; js < n_sw; ++js) {
            if (!__all_sync(0xffffffffu, mbar_wait(bar(9 + t), (n_tiles + js) & 1, abort_flag))) break;
            tc_fence_after();
            float sum = 0.f;
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                if (!((nz >> c) & 1u)) continue;
                float v[32];
                tc_ld32(tS + c * 32, v);
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const float2 mw = s_tab[t * 128 + c * 32 + e];
                    sum += fast_exp2(fmaf(v[e], a.scale_log2e, -mw.x)) * mw.y;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(19 + t));
            const int key = (sw0 + js) * 128 + row, jrel = key - a.affix_start;
            if (jrel >= 0 && jrel < a.affix_len)
                a.score_partial[(((int64_t)b * a.n_heads + h) * a.q_tiles + qt * 2 + t) * a.affix_len + jrel] = sum;
        }
      }
    }
    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) {
            atomicOr(a.status, kFlagWaitExpired);
            for (int i = 0; i < 4096; ++i) __nanosleep(64);   // let copies already in flight land
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// ---- host side ------------------------------------------------------------------------------
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn3() {
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

}  // namespace

// bf16 [batch, rows, cols] with row stride = cols and the given batch stride (elements);
// box = 64 cols x 128 rows x 1, 128-byte swizzle, zero fill out of bounds.
struct Map3Key { const void* ptr; int rows, cols, batch; int64_t bstride; int box_rows; };
struct Map3Entry { Map3Key key; CUtensorMap map; };
constexpr int kMap3Cache = 1024;
std::mutex g_map3_mutex;   // guards the cache below; a returned pointer is only good until the next lookup: callers copy the map
Map3Entry g_maps3[kMap3Cache];
int g_map3_count = 0, g_map3_next = 0;

const CUtensorMap* get_map3(const void* ptr, int rows, int cols, int batch, int64_t bstride, int box_rows) {
    for (int i = 0; i < g_map3_count; ++i) {
        const Map3Key& k = g_maps3[i].key;
        if (k.ptr == ptr && k.rows == rows && k.cols == cols && k.batch == batch && k.bstride == bstride && k.box_rows == box_rows)
            return &g_maps3[i].map;
    }
    EncodeTiledFn fn = encode_fn3();
    if (!fn) return nullptr;
    Map3Entry& e = g_maps3[g_map3_next];
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch};
    cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)bstride * 2};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    if (fn(&e.map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return nullptr;
    e.key = Map3Key{ptr, rows, cols, batch, bstride, box_rows};
    g_map3_next = (g_map3_next + 1) % kMap3Cache;
    if (g_map3_count < kMap3Cache) ++g_map3_count;
    return &e.map;
}

// Returns the number of kernels launched, 0 if this problem is not for the tensor-core kernel
// (the caller then uses the mma.sync kernel), -1 if a launch failed.
int launch_attention_tc(const AttnArgs& a, uint32_t* status, cudaStream_t stream) {
    if (a.head_dim != 128 || a.batch == 0 || a.n == 0) return 0;
    // reads through the position -> row map become two key sources when the key masks came with it
    const bool two_src = a.slot && a.pos_excl && a.row_keep && a.k_new && a.v_new;
    if (a.slot && !two_src) return 0;
    const int q_tiles = (a.n + 127) / 128;
    // measured at batch 1 with 26-4096 rows over 600-8300 keys: never slower than the key-split mma.sync
    // kernel, even with a single query tile per head (32 CTAs)
    static const int min_ctas = [] { const char* e = getenv("ACACHE_ATTN_TC_MIN_CTAS"); return e ? atoi(e) : 1; }();
    if ((int64_t)q_tiles * a.n_heads * a.batch < min_ctas) return 0;
    if ((a.kv_batch_stride * 2) % 16) return 0;
    const bool shared = a.kv_batch_stride == 0;           // one cache for the whole batch
    const int kv_cols = a.n_kv_heads * 128;
    std::lock_guard<std::mutex> lock(g_map3_mutex);
    // decode passes over a shared cache: the rows of several requests share one query tile (attention_group_kernel)
    static const bool group_on = [] { const char* e = getenv("ACACHE_ATTN_GROUP"); return !e || atoi(e) != 0; }();
    // Two requests of up to 64 rows where that saves rounds of CTAs.  A pair takes 1 to 5 % longer than one request, and half as many
    // rounds are less from two on, except two against two.  One | two to a tile, us, 48 rows, 32 heads, 2048 shared keys and 64 to 500
    // private rows per request: 7 requests (2 rounds | 1) 71-91 | 46-60, 9 (2 | 2) 73-94 | 75-95, 10 (3 | 2) 102-129 | 77-105,
    // 13 (3 | 2) 104-134 | 80-108, 19 (5 | 3) 172-218 | 121-161; 4096 shared keys, 9 requests 117 | 122; 28 heads, 9 (2 | 1) 111 | 66.
    const bool grouped = group_on && two_src && shared && a.batch >= 2;
    auto rounds = [&](int requests) { return ((a.batch + requests - 1) / requests * a.n_heads + sm_count() - 1) / sm_count(); };
    const int group = grouped && a.n <= 32 ? 4 : grouped && a.n <= 64 && rounds(2) < rounds(1) ? 2 : 1;
    CUtensorMap maps[5];
    const CUtensorMap* found[5];
    found[0] = get_map3(a.q, a.n, a.n_heads * 128, a.batch, (int64_t)a.n * a.n_heads * 128, 128 / group);
    if (found[0]) maps[0] = *found[0];
    found[1] = get_map3(a.cache_k, a.ctx_len, kv_cols, shared ? 1 : a.batch, shared ? (int64_t)a.ctx_len * kv_cols : a.kv_batch_stride);
    if (found[1]) maps[1] = *found[1];
    found[2] = get_map3(a.cache_v, a.ctx_len, kv_cols, shared ? 1 : a.batch, shared ? (int64_t)a.ctx_len * kv_cols : a.kv_batch_stride);
    if (found[2]) maps[2] = *found[2];
    const int n_fresh = a.n_fresh ? a.n_fresh : a.n;
    found[3] = two_src ? get_map3(a.k_new, n_fresh, kv_cols, a.batch, (int64_t)n_fresh * kv_cols) : found[1];
    if (found[3]) maps[3] = two_src ? *found[3] : maps[1];
    found[4] = two_src ? get_map3(a.v_new, n_fresh, kv_cols, a.batch, (int64_t)n_fresh * kv_cols) : found[2];
    if (found[4]) maps[4] = two_src ? *found[4] : maps[2];
    const CUtensorMap *mq = found[0] ? &maps[0] : nullptr, *mk = found[1] ? &maps[1] : nullptr, *mv = found[2] ? &maps[2] : nullptr,
                      *mkn = found[3] ? &maps[3] : nullptr, *mvn = found[4] ? &maps[4] : nullptr;
    if (!mq || !mk || !mv || !mkn || !mvn) return 0;
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(attention_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, AT_SMEM);
        cudaFuncSetAttribute(attention_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, AT_SMEM);
        cudaFuncSetAttribute(attention_tc2q_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AT2_SMEM);
        cudaFuncSetAttribute(attention_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AG_SMEM);
        attr = true;
    }
    AttnTcArgs t{};
    t.o = a.o; t.n = a.n; t.ctx_len = a.ctx_len; t.n_heads = a.n_heads; t.n_kv_heads = a.n_kv_heads;
    t.scale_log2e = 1.4426950408889634f / sqrtf(128.f);
    t.status = status;
    t.cache_shared = shared ? 1 : 0;
    t.group = group; t.batch = a.batch; t.q_tiles = q_tiles;
    if (two_src) {
        t.n_fresh_tiles = (n_fresh + 127) / 128; t.excl_words = a.excl_words; t.keep_words = a.keep_words;
        t.pos_excl = a.pos_excl; t.row_keep = a.row_keep;      // with key_drop the caller has OR-ed it into pos_excl
    } else if (a.key_drop) {
        t.excl_words = a.excl_words; t.pos_excl = a.key_drop;
    }
    t.kv_prefetch = 2;        // K/V tiles requested into L2 this many iterations ahead of the two-stage rings
    // Two query tiles per CTA pay off when the halved grid still fills the SMs and the context is short enough
    // for the per-CTA prologue and epilogue to matter (measured, one against the other: 2048-2560 keys with
    // 1000+ rows, 8-15 % faster; 8192 keys, 5-10 % slower; fewer CTAs than SMs, up to 1.8x slower).
    // ACACHE_ATTN_TC2Q = 0: never, 2: whenever there are two tiles.
    static const int mode_2q = [] { const char* e = getenv("ACACHE_ATTN_TC2Q"); return e ? atoi(e) : 1; }();
    const bool fused_score = a.score_rowmask && a.score_partial && group == 1;
    if (fused_score) {
        t.score_rowmask = a.score_rowmask; t.score_partial = a.score_partial; t.rm_words = a.rm_words;
        t.affix_start = a.affix_start; t.affix_len = a.affix_len; t.score_norm_full = a.score_norm_full;
    }
    // the scores are taken from the logits in the two-query-tile kernel only
    const bool use_2q = fused_score || mode_2q == 2 || (mode_2q == 1 && a.ctx_len + (two_src ? n_fresh : 0) <= 4096 &&
                                                        (int64_t)((q_tiles + 1) / 2) * a.n_heads * a.batch >= 148);
    cudaError_t err;
    if (use_2q && (q_tiles >= 2 || fused_score)) {
        err = launch_pdl(attention_tc2q_kernel, dim3((q_tiles + 1) / 2, a.n_heads, a.batch), dim3(AT2_THREADS), AT2_SMEM, stream, t,
                         *mq, *mk, *mv, *mkn, *mvn);
    } else {
        // Few query tiles leave most SMs idle, and one SM pulls K and V at 60-100 GB/s: the key tiles of a query tile are split
        // over a cluster of up to eight CTAs, as many as one wave holds while each still has two tiles.  Layer-step of 103 rows
        // over 1024 keys (32 query tiles): attention 17.3 -> 13.6 us with four CTAs, the step 153.5 us with one, 152.1 with
        // two, 150.0 with four; decode pass of 32 rows (4 layers) 679, 675, 665.
        const int groups = (a.batch + group - 1) / group;
        const int64_t ctas = (int64_t)q_tiles * a.n_heads * groups;
        const int tiles = (a.ctx_len + 127) / 128 + t.n_fresh_tiles * (a.batch - (groups - 1) * group);   // of the last group
        t.split = 1;
        while (t.split < 8 && ctas * t.split * 2 <= 148 && tiles >= t.split * 4) t.split *= 2;
        cudaLaunchConfig_t cfg{};
        t.n_items = (int)ctas;
        // from six rounds of CTAs on, items share a CTA (of the layer-step, 0.7-1.0 % at 13.8 rounds, 0.2-0.5 % at 8.6, 0.4-1.0 % at
        // 6.5; at 1.9 and 2.8 rounds, where the hardware's assignment evens out the last round, 0.3 and 0.9 % slower)
        const bool many = t.split == 1 && group == 1 && t.n_items >= 6 * sm_count();
        cfg.gridDim = dim3(many ? sm_count() : t.n_items * t.split);
        cfg.blockDim = dim3(AT_THREADS);
        cfg.dynamicSmemBytes = group > 1 ? AG_SMEM : AT_SMEM;
        cfg.stream = stream;
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        at[1].id = cudaLaunchAttributeClusterDimension;
        at[1].val.clusterDim.x = t.split; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = t.split > 1 ? 2 : 1;
        err = cudaLaunchKernelEx(&cfg, group > 1 ? attention_group_kernel : many ? attention_tc_kernel<true> : attention_tc_kernel<false>, t, *mq,
                                 *mk, *mv, *mkn, *mvn);
    }
    return err == cudaSuccess ? 1 : -1;
}

}  // namespace acache
