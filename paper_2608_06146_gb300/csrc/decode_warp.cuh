// decode_warp.cuh -- C2/C5: the warp path of one decode step, over either pool: the decode grid's CTAs run
// it after their tensor-core pieces, or from the start where they have none (decode_tc.cu).
//
// Every warp owns one work item and runs on its own: a 3-deep ring of 16-token
// paged blocks fetched with cp.async (each lane copies 16 of the block's 512 16-byte chunks into
// a 128-byte-swizzled [16][64] panel per half of K and V), one cp.async group per block, so no
// warp ever waits for another. cp.async rather than TMA: a 16-token block is only four 2 KB
// boxes, and an SM issues a TMA box only every ~70 cycles. The math puts the 8 query heads of a KV head
// in the N = 8 columns of mma.m16n8k16 and the 16 tokens of a block in its M = 16 rows:
//     S^T[16 tok x 8 heads] = K[16 x 128] . Q^T[128 x 8]             (8 MMAs)
//     O^T[128 x 8 heads]   += V^T[128 x 16 tok] . P^T[16 tok x 8]    (8 MMAs)
// so no MMA lane is padding. The P^T operand is the score fragment transposed in registers with
// movmatrix; the online softmax runs per head over the token axis with shuffles.
#pragma once

#include <float.h>
#include <math.h>

#include "common.cuh"
#include "tc.cuh"

namespace padoc_warp {

constexpr int kD = 128;          // head_dim of the bf16 path
constexpr int kGroup = 8;        // query heads per KV head of the bf16 path
constexpr int kBlk = 16;         // tokens per paged block
constexpr int kWarps = PADOC_WARP_KERNEL_WARPS;   // independent warps per CTA
constexpr int kWStages = 3;            // paged blocks in flight per warp
constexpr int kBoxBytes = kBlk * 128;  // one 16-row x 64-column box
constexpr int kWStageBytes = 4 * kBoxBytes;   // K lo, K hi, V lo, V hi
constexpr int kWarpRing = kWStages * kWStageBytes;
// E4M3 pool: a stage holds a block's K and V codes ([16 rows][128 bytes] each, 16-byte chunks
// swizzled by row) and its two scales. Half the bytes a block: six stages keep as much in flight.
constexpr int kE8Stages = 6;
constexpr int kE8Rows = kBlk * 128;                  // 2 KB of codes per tensor
constexpr int kE8StageBytes = 2 * kE8Rows + 128;     // K codes, V codes, scales (k, v)
constexpr int kE8WarpBytes = kE8Stages * kE8StageBytes;
// shared memory of the kWarps warps' rings, from a 1024-byte-aligned base
constexpr size_t kRingBytes = (size_t)kWarps * kWarpRing;
constexpr size_t kRingBytesE4M3 = (size_t)kWarps * kE8WarpBytes;

struct DecodeParams {
    const int32_t *stream_page, *shared_len, *private_len, *slot_ptr;
    const int32_t *page_len;     // each page's shared-stream length (the plan's)
    // 1: the previous kernel in the stream is this step's append (padoc_mpd_launch_step), which
    // writes only each stream's newest row and the step's queries: warps of CTAs without
    // tensor-core work read their headers and block ids and start their first blocks (those
    // without a newest row) before they wait for it
    int32_t pre_wait;
    // with pre_wait (may be null): [num_warps][4] pool rows of the first four blocks of each warp's
    // first item (-2 - row: the block of its stream's newest row; -1 past its end), read beside the
    // item header instead of after it
    const int32_t *first_blocks;
    const padoc_item *items;
    int32_t first_item;          // warp items start here
    const int32_t *warp_ptr;     // warp w owns warp items [warp_ptr[w], warp_ptr[w+1])
    int32_t num_warps;
    const int32_t *page_table;
    const int32_t *stream_table;
    int32_t page_stride, stream_stride;
    int32_t num_blocks, num_kv_heads, num_q_heads, pool_rows;
    const __nv_bfloat16 *k_pool, *v_pool;
    const uint8_t *k_codes, *v_codes;     // E4M3 pool (k_pool / v_pool unused)
    const float *k_scales, *v_scales;
    const __nv_bfloat16 *q;
    __nv_bfloat16 *part_o;       // partial O, bf16 (workspace layout in plan_internal.h)
    float *part_lse;
    float scale_log2;
    int *err;
};

// One warp of the warp path: warp `warp` of its CTA (its ring starts at smem + warp x the ring
// size; smem is 1024-byte aligned) runs warp list wi < prm.num_warps, whole warp, no CTA barrier.
// kPreWait: the CTA has not waited for the previous kernel in the stream (prm.pre_wait): the warp
// waits itself once its first safe blocks are on the way.
template <bool kE4M3, bool kPreWait = false>
__device__ __forceinline__ void decode_warp_role(const DecodeParams &prm, uint8_t *smem, int warp, int lane, int wi)
{
    uint8_t *wbuf = smem + (size_t)warp * (kE4M3 ? kE8WarpBytes : kWarpRing);
    constexpr int kStages = kE4M3 ? kE8Stages : kWStages;
    const padoc_item *items = prm.items + prm.first_item;
    const int i0 = prm.warp_ptr[wi], i1 = prm.warp_ptr[wi + 1];
    // Every global read the loop depends on is issued at least one item ahead: item headers two
    // items ahead, block ids (one per lane) and query fragments one item ahead, so a warp never
    // waits on a load between two paged blocks.
    auto load_item = [&](int u) { return items[u]; };   // 4-byte loads: the blob has no 16-byte alignment
    struct Walk {   // what the producer needs of an item
        const int32_t *table;
        int blk0, nblk, g;
        int rows;   // E4M3: from blk0's first on, those the item sees
    };
    auto walk_of = [&](const padoc_item &it) {
        Walk w;
        w.table = it.kind == PADOC_ITEM_SHARED ? prm.page_table + (size_t)it.index * prm.page_stride
                                               : prm.stream_table + (size_t)it.first_stream * prm.stream_stride;
        w.blk0 = it.tok_begin / kBlk;
        w.nblk = it.tok_end > it.tok_begin ? (it.tok_end - it.tok_begin + kBlk - 1) / kBlk : 0;
        w.g = it.kv_head;
        w.rows = it.tok_end - w.blk0 * kBlk;
        return w;
    };
    auto ids_of = [&](const Walk &w) { return lane < w.nblk ? w.table[w.blk0 + lane] : 0; };

    // The warp walks its items with one ring of kStages paged blocks that runs on from one item
    // into the next. Producer: the next block to fetch is block pb of item pu (walk pc, ids ids_c);
    // item pu + 1 (walk pn, ids ids_n) and the header of item pu + 2 (hn2) are already on the way.
    // kPreWait with first_blocks: lane k < 4 holds the pool row of block k of the first item (>= 0),
    // -2 - that row for the block holding its stream's newest row, -1 past the item's end
    const bool have_fb = kPreWait && prm.first_blocks != nullptr;
    const int32_t fb = have_fb && lane < 4 ? prm.first_blocks[(size_t)wi * 4 + lane] : -1;
    int pu = i0, pb = 0;
    Walk pc{prm.page_table, 0, 0, 0, 0}, pn{prm.page_table, 0, 0, 0, 0};
    int32_t ids_c = 0, ids_n = 0;
    padoc_item hn2 = {};
    if (i0 < i1) { pc = walk_of(load_item(i0)); ids_c = ids_of(pc); }
    if (i0 + 1 < i1) { pn = walk_of(load_item(i0 + 1)); ids_n = ids_of(pn); }
    if (i0 + 2 < i1) hn2 = load_item(i0 + 2);
    const uint64_t kv_policy = l2_evict_first_policy();   // paged blocks are read once per call
    int ring = 0;   // blocks issued so far: block n goes to stage n % kWStages
    // chunk q = lane + 32k of a block's 512 16-byte chunks is panel q / 128 (K lo, K hi, V lo, V hi),
    // row (q / 8) % 16, 16-byte column q % 8 (swizzled)
    auto issue_next = [&]() {   // whole warp; always commits a group, possibly empty
        while (pu < i1 && pb >= pc.nblk) {
            ++pu;
            pb = 0;
            pc = pn;
            ids_c = ids_n;
            if (pu + 1 < i1) { pn = walk_of(hn2); ids_n = ids_of(pn); }
            if (pu + 2 < i1) hn2 = load_item(pu + 2);
        }
        if (pu < i1) {
            // block ids past the 32 a warp holds are read directly (the planner keeps items shorter)
            const int32_t id = pb < 32 ? __shfl_sync(0xffffffffu, ids_c, pb) : pc.table[pc.blk0 + pb];
            const bool okid = id >= 0 && id < prm.num_blocks;
            if (!okid && lane == 0) padoc_record_error(prm.err, PADOC_DEVERR_BLOCK_ID, id);
            const size_t rowbase = okid ? ((size_t)id * prm.num_kv_heads + pc.g) * kBlk : 0;
            if constexpr (kE4M3) {
                // chunk q = lane + 32k of the block's 256 16-byte chunks of codes: tensor q / 128,
                // row (q / 8) % 16, chunk q % 8 (swizzled by row); lanes 0 and 1 also copy the K and
                // V scales of the (block, KV head) (zeros for a bad id, whose codes are zeros too). V rows
                // past the item's end land as zeros: a former owner's may hold NaN codes, against P = 0.
                const uint32_t base = smem_u32(wbuf + (ring % kStages) * kE8StageBytes);
                const int left = pc.rows - pb * kBlk;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int q = lane + 32 * k;
                    const int tn = q >> 7, r = (q >> 3) & 15, cc = q & 7;
                    const uint8_t *src = (tn == 0 ? prm.k_codes : prm.v_codes) + (rowbase + r) * kD + cc * 16;
                    cp_async_16_hint(base + tn * kE8Rows + r * 128 + ((cc ^ (r & 7)) << 4), src,
                                     okid && (tn == 0 || r < left) ? 16u : 0u, kv_policy);
                }
                if (lane < 2) {
                    const size_t si = okid ? (size_t)id * prm.num_kv_heads + pc.g : 0;
                    cp_async_4(base + 2 * kE8Rows + lane * 4, (lane == 0 ? prm.k_scales : prm.v_scales) + si,
                               okid ? 4u : 0u);
                }
            } else {
                const uint32_t base = smem_u32(wbuf + (ring % kStages) * kWStageBytes);
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const int q = lane + 32 * k;
                    const int panel = q >> 7, r = (q >> 3) & 15, cc = q & 7;
                    const __nv_bfloat16 *src = (panel < 2 ? prm.k_pool : prm.v_pool) +
                                               (rowbase + r) * kD + (panel & 1) * 64 + cc * 8;
                    cp_async_16_hint(base + panel * kBoxBytes + r * 128 + ((cc ^ (r & 7)) << 4), src, okid ? 16u : 0u,
                                     kv_policy);
                }
            }
            ++pb;
            ++ring;
        }
        cp_async_commit();
    };
    int pre = 0;
    if constexpr (kPreWait) {
        // Before the wait: the first item's blocks ahead of the block holding its stream's newest
        // row (page_len - 1 of a shared item's page, private_len - 1 of a private item's stream),
        // which the append may be writing; everything read so far (plan, block tables) was copied
        // before the append started.
        if (have_fb) {
            // straight from the rows the host wrote, without waiting for the item header: the
            // leading blocks that exist, are in the pool and hold no newest row
            const bool ok = lane < 4 && fb >= 0 && fb <= prm.pool_rows - kBlk;
            const uint32_t okm = __ballot_sync(0xffffffffu, ok) & 0xfu;
            pre = min(__ffs(~okm) - 1, kWStages);
            for (int k = 0; k < pre; ++k) {
                const size_t rowbase = (size_t)__shfl_sync(0xffffffffu, fb, k);
                const uint32_t base = smem_u32(wbuf + k * kWStageBytes);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const int q = lane + 32 * c;
                    const int panel = q >> 7, r = (q >> 3) & 15, cc = q & 7;
                    const __nv_bfloat16 *src = (panel < 2 ? prm.k_pool : prm.v_pool) +
                                               (rowbase + r) * kD + (panel & 1) * 64 + cc * 8;
                    cp_async_16_hint(base + panel * kBoxBytes + r * 128 + ((cc ^ (r & 7)) << 4), src, 16u, kv_policy);
                }
                cp_async_commit();
            }
            pb = pre;
            ring = pre;
        } else if (i0 < i1) {
            const padoc_item it0 = load_item(i0);
            const int32_t len = it0.kind == PADOC_ITEM_SHARED ? prm.page_len[it0.index] : prm.private_len[it0.first_stream];
            pre = min(min(kWStages, pc.nblk), max(0, (len - 1) / kBlk - pc.blk0));
            for (int k = 0; k < pre; ++k) issue_next();
        }
        pdl_wait_prerequisite();
        pdl_launch_dependents();
    }
    for (int k = pre; k < kStages; ++k) issue_next();

    // Consumer: header of the next item (ch_n) and of the one after (ch_n2), and the next item's
    // query fragments (B operand Q^T[128 dims x 8 heads]) and first partial row.
    padoc_item ch_n = {}, ch_n2 = {};
    uint32_t qn[8][2];
    size_t row_n = 0;
    auto load_q = [&](const padoc_item &it) {
        const __nv_bfloat16 *qrow =
            prm.q + ((size_t)it.first_stream * prm.num_q_heads + it.kv_head * kGroup + (lane >> 2)) * kD;
        if constexpr (kE4M3) {   // a lane's share of a row is 32 contiguous dims, four to a k-step (see below)
            const uint4 *src = reinterpret_cast<const uint4 *>(qrow + (lane & 3) * 32);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 x = src[c];
                qn[2 * c][0] = x.x; qn[2 * c][1] = x.y; qn[2 * c + 1][0] = x.z; qn[2 * c + 1][1] = x.w;
            }
        } else {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                qn[ks][0] = *reinterpret_cast<const uint32_t *>(qrow + ks * 16 + (lane & 3) * 2);
                qn[ks][1] = *reinterpret_cast<const uint32_t *>(qrow + ks * 16 + 8 + (lane & 3) * 2);
            }
        }
        row_n = (size_t)(prm.slot_ptr[(size_t)it.first_stream * prm.num_kv_heads + it.kv_head] + it.slot) * kGroup;
    };
    if (i0 < i1) { ch_n = load_item(i0); load_q(ch_n); }
    if (i0 + 1 < i1) ch_n2 = load_item(i0 + 1);
    int gc = 0;   // blocks consumed so far
    for (int cu = i0; cu < i1; ++cu) {
        const padoc_item it = ch_n;
        uint32_t qb[8][2];
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) { qb[ks][0] = qn[ks][0]; qb[ks][1] = qn[ks][1]; }
        const size_t row0 = row_n;
        if (cu + 1 < i1) {
            ch_n = ch_n2;
            load_q(ch_n);
            if (cu + 2 < i1) ch_n2 = load_item(cu + 2);
        }
        const int cutoff = it.tok_end;   // the planner keeps warp items inside their stream's cutoff
        const int blk0 = it.tok_begin / kBlk;
        const int nblk = cutoff > it.tok_begin ? (cutoff - it.tok_begin + kBlk - 1) / kBlk : 0;
        float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};   // heads h0 = 2*(lane%4), h0+1
        // E4M3: the queries as f16, their scale off again in the score multipliers of heads h0, h0 + 1; mv: the
        // maxima of score + log2 of the V scale, which P is taken against (m: of the scores, for the row sums)
        float qk0 = prm.scale_log2, qk1 = prm.scale_log2;
        float mv[2] = {-INFINITY, -INFINITY};
        if constexpr (kE4M3) {
            float amax = 0.f, qs, qi;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) amax = bf16x2_amax(bf16x2_amax(amax, qb[ks][0]), qb[ks][1]);
            amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
            amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
            f16_row_scale(amax, qs, qi);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                qb[ks][0] = bf16x2_to_f16x2(qb[ks][0], qs);
                qb[ks][1] = bf16x2_to_f16x2(qb[ks][1], qs);
            }
            qk0 *= __shfl_sync(0xffffffffu, qi, 8 * (lane & 3));
            qk1 *= __shfl_sync(0xffffffffu, qi, 8 * (lane & 3) + 4);
        }
        float o[8][4];
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f;

        if constexpr (kE4M3) {
            // The MMAs' operands come straight from the codes. The order of a contraction's elements is free
            // as long as both operands share it, so k-step ks of S^T takes dims 32 j + 4 ks .. + 3 of lane
            // j = lane % 4 (its rows' 32 contiguous bytes), and M row (m, half) of m-tile mt of O^T is dim
            // 16 m + 2 mt + half (16 contiguous bytes of each of its four tokens, two tokens' bytes
            // interleaved into pairs): one conversion instruction per two values, exact in f16, and no
            // expanded copy in shared memory. The serving batch's lists alone: 52 us with the copy, 36 us so
            // (with two or three blocks to a turn of the softmax 38 and 41 us).
            const int r = lane >> 2, j = lane & 3;
            auto word = [](const uint4 &v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; };
            for (int bi = 0; bi < nblk; ++bi, ++gc) {
                cp_async_wait<kStages - 1>();   // block gc has landed (one group per block)
                __syncwarp();
                const uint8_t *stg = wbuf + (gc % kStages) * kE8StageBytes;
                const float ks = *reinterpret_cast<const float *>(stg + 2 * kE8Rows);
                const float vs = *reinterpret_cast<const float *>(stg + 2 * kE8Rows + 4);
                uint4 kc[2][2], vc[4];
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh)
                        kc[c][hh] = *reinterpret_cast<const uint4 *>(stg + (r + 8 * hh) * 128 + (((2 * j + c) ^ r) << 4));
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int t = 2 * j + (c & 1) + 8 * (c >> 1);
                    vc[c] = *reinterpret_cast<const uint4 *>(stg + kE8Rows + t * 128 + ((r ^ (t & 7)) << 4));
                }
                // A zero scale marks a block without a nonzero value (its codes are zeros): any K factor gives its
                // scores, and its V counts nowhere. The V scale is 2^ev times a mantissa (NaN for none that is a
                // finite number), which with 2^6 rides on P.
                const bool tiny = vs < 0x1p-60f;
                const uint32_t vb = __float_as_uint(tiny ? vs * 0x1p64f : vs);
                const float ev = vs > 0.f ? (float)((int)(vb >> 23) - (tiny ? 127 + 64 : 127)) : -INFINITY;
                const float pf = !(vs <= FLT_MAX) ? NAN : vs > 0.f ? __uint_as_float((vb & 0x007FFFFFu) | 0x42800000u) : 0.f;
                const float kf = ks > 0.f ? ks : 1.f;
                const uint64_t km = f2_mul(f2_pack(qk0, qk1), f2_pack(kf, kf));
                __syncwarp();   // every lane has its part: the stage may be refilled
                issue_next();
                // S^T = K . Q^T, two independent MMA chains
                float acc[2][4];
#pragma unroll
                for (int c = 0; c < 2; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.f;
#pragma unroll
                for (int ks8 = 0; ks8 < 8; ++ks8) {
                    const uint32_t x0 = word(kc[ks8 >> 2][0], ks8 & 3), x1 = word(kc[ks8 >> 2][1], ks8 & 3);
                    const uint32_t a[4] = {e4m3x2_to_f16x2((uint16_t)x0), e4m3x2_to_f16x2((uint16_t)x1),
                                           e4m3x2_to_f16x2((uint16_t)(x0 >> 16)), e4m3x2_to_f16x2((uint16_t)(x1 >> 16))};
                    mma_f16_16816(acc[ks8 & 1], a, qb[ks8][0], qb[ks8][1]);
                }
                const int t0 = (blk0 + bi) * kBlk + r, t1 = t0 + 8;
                float s0, s1, s2, s3;
                f2_unpack(f2_mul(f2_add(f2_pack(acc[0][0], acc[0][1]), f2_pack(acc[1][0], acc[1][1])), km), s0, s1);
                f2_unpack(f2_mul(f2_add(f2_pack(acc[0][2], acc[0][3]), f2_pack(acc[1][2], acc[1][3])), km), s2, s3);
                if (t0 >= cutoff) s0 = s1 = -INFINITY;
                if (t1 >= cutoff) s2 = s3 = -INFINITY;
                float mx0 = fmaxf(s0, s2), mx1 = fmaxf(s1, s3);
#pragma unroll
                for (int sh = 4; sh < 32; sh <<= 1) {
                    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, sh));
                    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, sh));
                }
                const float mn0 = fmaxf(m[0], mx0), mn1 = fmaxf(m[1], mx1);
                const float vn0 = fmaxf(mv[0], mx0 + ev), vn1 = fmaxf(mv[1], mx1 + ev);
                if (__any_sync(0xffffffffu, mn0 != m[0] || mn1 != m[1] || vn0 != mv[0] || vn1 != mv[1])) {   // a maximum moved
                    // (what has only been masked, or weighed by zero scales, keeps -inf and holds zeros)
                    l[0] *= mn0 == -INFINITY ? 1.f : fast_exp2(m[0] - mn0);
                    l[1] *= mn1 == -INFINITY ? 1.f : fast_exp2(m[1] - mn1);
                    const float al0 = vn0 == -INFINITY ? 1.f : fast_exp2(mv[0] - vn0);
                    const float al1 = vn1 == -INFINITY ? 1.f : fast_exp2(mv[1] - vn1);
#pragma unroll
                    for (int mt = 0; mt < 8; ++mt) {
                        o[mt][0] *= al0; o[mt][1] *= al1; o[mt][2] *= al0; o[mt][3] *= al1;
                    }
                    m[0] = mn0; m[1] = mn1;
                    mv[0] = vn0; mv[1] = vn1;
                }
                // P is the probability times 2^f, f = V scale over the largest weighted one, at most 1; where f would
                // be below -60 (0 in f16 either way) it is -60, and P times 2^-f is the probability for the row sum
                const float r0 = mn0 == -INFINITY ? 0.f : mn0, r1 = mn1 == -INFINITY ? 0.f : mn1;
                const float f0 = fmaxf(ev + (r0 - (vn0 == -INFINITY ? INFINITY : vn0)), -60.f);
                const float f1 = fmaxf(ev + (r1 - (vn1 == -INFINITY ? INFINITY : vn1)), -60.f);
                const uint64_t fr = f2_sub(f2_pack(f0, f1), f2_pack(r0, r1)), pf2 = f2_pack(pf, pf);
                float x0, x1, x2, x3, y0, y1, y2, y3;
                f2_unpack(f2_add(f2_pack(s0, s1), fr), x0, x1);
                f2_unpack(f2_add(f2_pack(s2, s3), fr), x2, x3);
                const uint64_t p01 = f2_pack(fast_exp2(x0), fast_exp2(x1)), p23 = f2_pack(fast_exp2(x2), fast_exp2(x3));
                f2_unpack(f2_fma(f2_add(p01, p23), f2_pack(fast_exp2(-f0), fast_exp2(-f1)), f2_pack(l[0], l[1])), l[0], l[1]);
                f2_unpack(f2_mul(p01, pf2), y0, y1);
                f2_unpack(f2_mul(p23, pf2), y2, y3);
                const uint32_t b0 = movmatrix_trans(pack_f16x2(y0, y1)), b1 = movmatrix_trans(pack_f16x2(y2, y3));
#pragma unroll
                for (int w = 0; w < 4; ++w)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {   // dims 4 w + 2 hh, + 1 of the lane's 16
                        const uint32_t lo = __byte_perm(word(vc[0], w), word(vc[1], w), hh ? 0x7362 : 0x5140);
                        const uint32_t hi = __byte_perm(word(vc[2], w), word(vc[3], w), hh ? 0x7362 : 0x5140);
                        const uint32_t a[4] = {e4m3x2_to_f16x2((uint16_t)lo), e4m3x2_to_f16x2((uint16_t)(lo >> 16)),
                                               e4m3x2_to_f16x2((uint16_t)hi), e4m3x2_to_f16x2((uint16_t)(hi >> 16))};
                        mma_f16_16816(o[2 * w + hh], a, b0, b1);
                    }
            }
        } else {
            for (int bi = 0; bi < nblk; ++bi, ++gc) {
                cp_async_wait<kStages - 1>();   // block gc has landed (one group per block)
                __syncwarp();
                const uint32_t base = smem_u32(wbuf + (gc % kStages) * kWStageBytes);
                const int tokbase = (blk0 + bi) * kBlk;
                // S^T = K . Q^T, as two independent MMA chains (even / odd k-steps) added at the end
                float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    const uint32_t row = lane & 15;
                    const uint32_t col = (ks & 3) * 16 + (lane >> 4) * 8;
                    uint32_t a[4];
                    ldmatrix_x4(a, base + (ks >> 2) * kBoxBytes + sw128_offset(row, col));
                    mma_bf16_16816((ks & 1) ? acc2 : acc, a, qb[ks][0], qb[ks][1]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] += acc2[i];
                const int t0 = tokbase + (lane >> 2), t1 = t0 + 8;
                float sc[4];
                sc[0] = t0 < cutoff ? acc[0] * prm.scale_log2 : -INFINITY;
                sc[1] = t0 < cutoff ? acc[1] * prm.scale_log2 : -INFINITY;
                sc[2] = t1 < cutoff ? acc[2] * prm.scale_log2 : -INFINITY;
                sc[3] = t1 < cutoff ? acc[3] * prm.scale_log2 : -INFINITY;
                float mx0 = fmaxf(sc[0], sc[2]), mx1 = fmaxf(sc[1], sc[3]);
#pragma unroll
                for (int sh = 4; sh < 32; sh <<= 1) {
                    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, sh));
                    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, sh));
                }
                const float mn0 = fmaxf(m[0], mx0), mn1 = fmaxf(m[1], mx1);
                // a head whose columns are all masked so far keeps m = -inf and contributes 0
                const float al0 = mn0 == -INFINITY ? 1.f : fast_exp2(m[0] - mn0);
                const float al1 = mn1 == -INFINITY ? 1.f : fast_exp2(m[1] - mn1);
                const float r0 = mn0 == -INFINITY ? 0.f : mn0, r1 = mn1 == -INFINITY ? 0.f : mn1;
                const float p0 = fast_exp2(sc[0] - r0), p1 = fast_exp2(sc[1] - r1);
                const float p2 = fast_exp2(sc[2] - r0), p3 = fast_exp2(sc[3] - r1);
                m[0] = mn0; m[1] = mn1;
                l[0] = l[0] * al0 + p0 + p2;
                l[1] = l[1] * al1 + p1 + p3;
                const uint32_t b0 = movmatrix_trans(pack_bf16x2(p0, p1));
                const uint32_t b1 = movmatrix_trans(pack_bf16x2(p2, p3));
                if (__any_sync(0xffffffffu, al0 != 1.f || al1 != 1.f)) {   // a head's running max moved
#pragma unroll
                    for (int mt = 0; mt < 8; ++mt) {
                        o[mt][0] *= al0; o[mt][1] *= al1; o[mt][2] *= al0; o[mt][3] *= al1;
                    }
                }
#pragma unroll
                for (int mt = 0; mt < 8; ++mt) {
                    const int i = lane >> 3;
                    const uint32_t row = (lane & 7) + (i >= 2 ? 8 : 0);
                    const uint32_t col = (mt & 3) * 16 + (i & 1) * 8;
                    uint32_t a[4];
                    ldmatrix_x4_trans(a, base + (2 + (mt >> 2)) * kBoxBytes + sw128_offset(row, col));
                    mma_bf16_16816(o[mt], a, b0, b1);
                }
                __syncwarp();   // every lane is done with the stage
                issue_next();
            }
        }
        // complete the row sums over the 8 token lanes of each head
#pragma unroll
        for (int sh = 4; sh < 32; sh <<= 1) {
            l[0] += __shfl_xor_sync(0xffffffffu, l[0], sh);
            l[1] += __shfl_xor_sync(0xffffffffu, l[1], sh);
        }
        // the partial in bf16, in the slot layout [16 chunks of 8 dims][8 heads][8]: lane l holds dim
        // l / 4 of heads h0, h0 + 1 (h0 = 2 (l % 4)); with its partner l ^ 4 (the next or previous dim)
        // a lane of an even dim writes the dim pair of head h0, one of an odd dim that of head
        // h0 + 1, so that the warp writes each chunk's [8 heads][8 dims] as one 128-byte run
        if constexpr (kE4M3) {
            // a lane holds dims 16 (l / 4) .. + 15 of both heads: two 16-byte pieces of each
            const int h0 = (lane & 3) * 2;
            // (in two factors: with V scales near the ends of fp32's range their product leaves it)
            const float i0f = l[0] > 0.f ? 1.f / l[0] : 0.f, i1f = l[1] > 0.f ? 1.f / l[1] : 0.f;
            const float e0f = mv[0] == -INFINITY ? 0.f : exp2f(mv[0] - 6.f - m[0]);
            const float e1f = mv[1] == -INFINITY ? 0.f : exp2f(mv[1] - 6.f - m[1]);
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
                o[mt][0] = o[mt][0] * i0f * e0f; o[mt][1] = o[mt][1] * i1f * e1f;
                o[mt][2] = o[mt][2] * i0f * e0f; o[mt][3] = o[mt][3] * i1f * e1f;
            }
            __nv_bfloat16 *p = prm.part_o + row0 * kD + (lane >> 2) * 128 + h0 * 8;   // chunk 2 (l / 4)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                *reinterpret_cast<uint4 *>(p + 64 * c) =
                    make_uint4(pack_bf16x2(o[4 * c][0], o[4 * c][2]), pack_bf16x2(o[4 * c + 1][0], o[4 * c + 1][2]),
                               pack_bf16x2(o[4 * c + 2][0], o[4 * c + 2][2]), pack_bf16x2(o[4 * c + 3][0], o[4 * c + 3][2]));
                *reinterpret_cast<uint4 *>(p + 64 * c + 8) =
                    make_uint4(pack_bf16x2(o[4 * c][1], o[4 * c][3]), pack_bf16x2(o[4 * c + 1][1], o[4 * c + 1][3]),
                               pack_bf16x2(o[4 * c + 2][1], o[4 * c + 2][3]), pack_bf16x2(o[4 * c + 3][1], o[4 * c + 3][3]));
            }
        } else {
            const int h0 = (lane & 3) * 2, dm = lane >> 2;
            const bool ev = (dm & 1) == 0;
            const float i0f = l[0] > 0.f ? 1.f / l[0] : 0.f, i1f = l[1] > 0.f ? 1.f / l[1] : 0.f;
            // element offset of this lane's pair inside a chunk
            const int off = ev ? h0 * 8 + dm : (h0 + 1) * 8 + dm - 1;
            uint32_t *p = reinterpret_cast<uint32_t *>(prm.part_o + row0 * kD);   // row0 = slot * 8
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {   // chunk 2 mt + c: registers 2c (head h0), 2c + 1 (h0 + 1)
                    const float a = o[mt][2 * c] * i0f, b = o[mt][2 * c + 1] * i1f;
                    const float pa = __shfl_xor_sync(0xffffffffu, a, 4), pb = __shfl_xor_sync(0xffffffffu, b, 4);
                    p[((2 * mt + c) * 64 + off) >> 1] = ev ? pack_bf16x2(a, pa) : pack_bf16x2(pb, b);
                }
            }
        }
        if (lane < 4) {
            const int h0 = lane * 2;
            prm.part_lse[row0 + h0] = l[0] > 0.f ? (m[0] + log2f(l[0])) * PADOC_LN2 : -INFINITY;
            prm.part_lse[row0 + h0 + 1] = l[1] > 0.f ? (m[1] + log2f(l[1])) * PADOC_LN2 : -INFINITY;
        }
    }
    cp_async_wait<0>();
}

}  // namespace padoc_warp
