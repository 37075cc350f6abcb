// prefill_bwd_tc.cu -- gradients of the packed ancestor prefill on the 5th-generation tensor cores
// (App. C.1: the backward of the tree-varlen attention; Sec. 3.2 visibility), in two passes that
// need neither a gather nor atomics.
//
// With c = scale * log2(e), lse2 = lse * log2(e) and D = rowsum(dO * O) per query row and head
// (-lse2 and D precomputed per head, [Hq][t_pad], padded rows -lse2 = -inf so that their P is 0):
//   P = exp2(S c - lse2),  dS = P (dP - D),  S = Q K^T,  dP = dO V^T.
//
// dK/dV pass: a unit is a (128-key k-tile, KV head), units taken in the key-major map's order (most
//   work first), run by a cluster of 1, 2, 4 or 8 CTAs that share out its steps and add their fp32 sums
//   through distributed shared memory (pick_cluster below). For every (64-row q-tile that sees the
//   k-tile, query head reading the KV head) step the tensor cores form S^T = K Q^T (K from shared
//   memory) and dP^T = V dO^T (V copied to tensor memory once), the softmax warps write P^T and dS^T
//   as bf16 over S^T, and dV += P^T dO, dK += dS^T Q accumulate in tensor memory over the whole walk.
//   Every query that sees a shared-stream key (the stream's later tokens and each branch forked after
//   it) therefore adds into that key's gradient inside one cluster: the scatter-add of the gather's
//   backward, with nothing scattered.
// dQ pass: a unit is a (128-row q-tile, query head), heavier q-tiles first; a running CTA takes over units
//   not yet launched (cluster launch control), and the next unit's loads and first scores come under the
//   last one's output. It walks the query-major map of 64-key k-tiles: S = Q K^T (Q in tensor memory),
//   dP = dO V^T (dO in shared memory), dS as bf16 over S, dQ += dS K.
//
// What bounds a step is less its MMAs (about 1150 cycles in the dK/dV pass, 900 in the dQ pass, of
// 1500 and 1000) than the chain S -> softmax -> accumulation -> S, whose hand-overs take 300 to 400 cycles
// each because a warp's wait queues up behind the MMAs it has issued. So:
// - S, dP and the accumulating MMAs are issued by a warp each;
// - P and dS share S's columns, so dP's buffer is free again as soon as it is read, and the room that
//   gives holds V (dK/dV pass) or a third S buffer (dQ pass);
// - waits and roles are uniform per warp (see mbar_wait_warp), and a step's map entry is read a step ahead.
// A packed batch of 34107 tokens, 16 query heads: dK/dV pass 735 -> 657 us; dQ pass 644 -> 490 us (of which
// 70 us are its tiles of Q, dO and O, copied by TMA: the rows read lane by lane took 8000 cycles a
// CTA), -> 440 us with units taken over (a unit's start and end were 8000 of its 35000 cycles). One page
// of 3419 tokens: both passes 161 -> 140 -> 137 us.
//
// A softmax warp owns 32 TMEM lanes (rows) and one 32-column half of a step. Its bf16 results go to the
// first 16 columns of its own half of S (dS of the dK/dV pass to the other 16), so no warp overwrites
// a column another warp still has to read.
//
// Warp roles (384 threads): warps 0-7 softmax and epilogue, warp 8 TMA producer, warp 9 TMEM allocation
// and S, warp 10 the accumulating MMAs, warp 11 dP (converged warps, one elected lane issues). Every
// wait is bounded; a wait that runs out records an error and all roles leave their loops, the MMA
// warps wait for their MMAs, the producer for its copies, and tensor memory is released.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "tc.cuh"

namespace {

constexpr int kD = 128;
constexpr int kThreads = 384;
constexpr uint32_t kTmemCols = 512;

struct BwdParams {
    const int32_t *spans, *ptr, *idx, *order;
    const int8_t *kind;
    float *lt, *dt;                     // [Hq][t_pad]: -lse2 and D (written by the dQ pass, read by the dK/dV pass)
    const float *lse;                   // the forward's log-sum-exp, natural log, [T][Hq]
    int64_t T, t_pad;
    int32_t num_q_heads, num_kv_heads, num_tiles;
    float scale_log2, scale;
    __nv_bfloat16 *out0, *out1;         // dK/dV pass: dK, dV
    int *err;
};

__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, int *err, int site, volatile int *abort_flag)
{
    if (*abort_flag) return false;
    if (mbar_wait_bounded(bar, parity, err, site)) return true;
    *abort_flag = 1;
    return false;
}

// TMEM column of k-slice k (16 values) of a W-wide bf16 operand written by the softmax warps: column
// half c packs its W/2 values into the first W/4 columns of its own half.
template <int W>
__host__ __device__ constexpr uint32_t slice_col(int k)
{
    constexpr int per_half = W / 32;
    return (uint32_t)((k / per_half) * (W / 2) + (k % per_half) * 8);
}

__device__ __forceinline__ void store_row_bf16(__nv_bfloat16 *dst, const float (&o)[16], float mul)
{
#pragma unroll
    for (int i = 0; i < 16; i += 8) {
        uint4 w;
        w.x = pack_bf16x2(o[i] * mul, o[i + 1] * mul);
        w.y = pack_bf16x2(o[i + 2] * mul, o[i + 3] * mul);
        w.z = pack_bf16x2(o[i + 4] * mul, o[i + 5] * mul);
        w.w = pack_bf16x2(o[i + 6] * mul, o[i + 7] * mul);
        *reinterpret_cast<uint4 *>(dst + i) = w;
    }
}
__device__ __forceinline__ int clamp_w(int x, int w) { return min(max(x, 0), w); }

// 32 x 32 bit-matrix transpose across a warp: lane r holds row r (bit c = element (r, c)); on return
// lane r holds column r (bit c = element (c, r)). Five exchange rounds, each swapping the off-diagonal
// j x j blocks between lanes r and r ^ j.
__device__ __forceinline__ uint32_t transpose32_warp(uint32_t x, int lane)
{
    uint32_t m = 0x0000FFFFu;
#pragma unroll
    for (int j = 16; j != 0; j >>= 1) {
        const uint32_t o = __shfl_xor_sync(0xffffffffu, x, j);
        if (lane & j) x ^= ((o >> j) ^ x) & m;
        else x ^= (((x >> j) ^ o) & m) << j;
        m ^= m << (j >> 1);
    }
    return x;
}

// ================================================================================================
// dK/dV pass
// ================================================================================================
namespace dkv {
constexpr int kKT = PADOC_BWD_DKV_K_TILE;   // 128 keys: the M of every MMA
constexpr int kQT = PADOC_BWD_DKV_Q_TILE;   // 64 queries per step
constexpr int kStages = 4;   // (3: the Q of the step after next is still on its way, +1.5% time)
constexpr uint32_t kColS = 0, kColDP = 128, kColV = 192, kColAcc0 = 256, kColAcc1 = 384;   // kColS: two buffers
constexpr int kKPanel = kKT * 128;           // [128 rows][64 bf16]
constexpr int kQPanel = kQT * 128;           // [64 rows][64 bf16]
constexpr int kKTile = 2 * kKPanel;
constexpr int kQTile = 2 * kQPanel;
constexpr int kAuxBytes = 2 * kQT * 4 + kQT * 16;   // lse2[64], D[64], spans[64][4]
enum {
    B_KV = 0,
    B_QFULL = 1,                  // [stage]
    B_QEMPTY = 1 + kStages,       // [stage]
    B_SFULL = 1 + 2 * kStages,    // [step parity]
    B_PFULL = 3 + 2 * kStages,    // [step parity], an arrival per softmax warp
    B_ACC = 5 + 2 * kStages,      // [step parity]: the step's accumulating MMAs are done
    B_DPFREE = 7 + 2 * kStages,   // dP is read (an arrival per softmax warp)
    B_VT = 8 + 2 * kStages,       // V is in tensor memory (an arrival per softmax warp)
    B_FINAL = 9 + 2 * kStages,    // [issuing warp]
    B_COUNT = 12 + 2 * kStages
};
constexpr size_t kSmemBytes = 1024 + 2 * (size_t)kKTile + 2 * (size_t)kStages * kQTile + (size_t)kStages * kAuxBytes +
                              B_COUNT * 8 + 64;
}  // namespace dkv

// NC: the CTAs of a unit's cluster.
template <int NC>
__global__ void __launch_bounds__(kThreads, 1)
prefill_bwd_dkv_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap gmap,
                       const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                       const BwdParams prm)
{
    using namespace dkv;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sk = smem;
    uint8_t *sv = sk + kKTile;
    uint8_t *sq = sv + kKTile;                 // [stage] Q step tiles
    uint8_t *sg = sq + kStages * kQTile;       // [stage] dO step tiles
    uint8_t *aux = sg + kStages * kQTile;      // [stage] lse2, D, spans
    uint64_t *bars = (uint64_t *)(aux + kStages * kAuxBytes);
    uint32_t *tmem_slot = (uint32_t *)(bars + B_COUNT);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (a value the compiler knows to be warp-uniform)
    const int hkv = prm.num_kv_heads, group = prm.num_q_heads / hkv;
    // the cluster's unit, and this CTA's steps of it: ub .. ub + nu - 1
    const int unit = (int)blockIdx.x / NC, rank = (int)blockIdx.x % NC, g = unit % hkv;
    const int kt = __shfl_sync(0xffffffffu, prm.order[unit / hkv], 0);
    const int e0 = __shfl_sync(0xffffffffu, prm.ptr[kt], 0), steps = (__shfl_sync(0xffffffffu, prm.ptr[kt + 1], 0) - e0) * group;
    const int ub = (int)((int64_t)steps * rank / NC), nu = (int)((int64_t)steps * (rank + 1) / NC) - ub;
    auto bar = [&](int i) { return smem_u32(&bars[i]); };

    if (tid == 0) {
        for (int i = 0; i < B_COUNT; ++i) mbar_init(bar(i), (i == B_PFULL || i == B_PFULL + 1 || i == B_DPFREE || i == B_VT) ? 8
                                                                  : i == B_SFULL || i == B_SFULL + 1 ? 2 : 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 9) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const int lq = warp & 3, ch = warp >> 2;          // softmax warps: TMEM lane quarter, column half
    const int key = kt * kKT + lq * 32 + lane;
    const uint32_t lanes = (uint32_t)(lq * 32) << 16;
    bool sums = false;                                // softmax warps: this CTA's dV and dK are complete

    if (warp == 8) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0 && nu == 0) pdl_wait_prerequisite();
        if (lane == 0 && nu > 0) {
            tma_prefetch_desc(&qmap);
            tma_prefetch_desc(&gmap);
            tma_prefetch_desc(&kmap);
            tma_prefetch_desc(&vmap);
            pdl_wait_prerequisite();   // -lse2 and D are the dQ pass's
            mbar_arrive_expect_tx(bar(B_KV), 2 * kKTile);
            tma_load_2d(smem_u32(sk), &kmap, g * kD, kt * kKT, bar(B_KV));
            tma_load_2d(smem_u32(sk) + kKPanel, &kmap, g * kD + 64, kt * kKT, bar(B_KV));
            tma_load_2d(smem_u32(sv), &vmap, g * kD, kt * kKT, bar(B_KV));
            tma_load_2d(smem_u32(sv) + kKPanel, &vmap, g * kD + 64, kt * kKT, bar(B_KV));
            int issued = 0;
            for (int u = 0; u < nu; ++u) {
                const int s = u % kStages;
                if (u >= kStages && !wait_or_abort(bar(B_QEMPTY + s), (u / kStages - 1) & 1, prm.err, 50, abort_flag))
                    break;
                const int e = e0 + (ub + u) / group, h = g * group + (ub + u) % group;
                const int q0 = prm.idx[e] * kQT;
                const int nsp = prm.kind[e] == PADOC_TILE_FULL ? 0 : min(kQT, (int)(prm.T - q0)) * 16;
                const uint32_t fb = bar(B_QFULL + s);
                const uint32_t qb = smem_u32(sq + s * kQTile), gb = smem_u32(sg + s * kQTile);
                const uint32_t ab = smem_u32(aux + s * kAuxBytes);
                mbar_arrive_expect_tx(fb, 2 * kQTile + 2 * kQT * 4 + nsp);
                tma_load_2d(qb, &qmap, h * kD, q0, fb);
                tma_load_2d(qb + kQPanel, &qmap, h * kD + 64, q0, fb);
                tma_load_2d(gb, &gmap, h * kD, q0, fb);
                tma_load_2d(gb + kQPanel, &gmap, h * kD + 64, q0, fb);
                bulk_load(ab, prm.lt + (size_t)h * prm.t_pad + q0, kQT * 4, fb);
                bulk_load(ab + kQT * 4, prm.dt + (size_t)h * prm.t_pad + q0, kQT * 4, fb);
                if (nsp) bulk_load(ab + 2 * kQT * 4, prm.spans + 4 * (size_t)q0, (uint32_t)nsp, fb);
                issued = u + 1;
            }
            // copies still in flight must land before the CTA's shared memory is released
            mbar_wait_bounded(bar(B_KV), 0, prm.err, 51);
            for (int u = (issued > kStages ? issued - kStages : 0); u < issued; ++u)
                mbar_wait_bounded(bar(B_QFULL + u % kStages), (u / kStages) & 1, prm.err, 52);
        }
    } else if (warp >= 9) {
        // ---------------------------------------------------------------- MMA issuers (whole warps)
        // Warp 9 S^T, warp 11 dP^T, warp 10 the accumulating MMAs: one's waits, each behind the MMAs it
        // has issued, leave the tensor cores the others' MMAs. A step's S^T waits for the accumulating
        // MMAs that read the buffer it overwrites, its dP^T for the softmax warps' reads of the last one.
        if (nu > 0) {
            auto wait_w = [&](int b, uint32_t parity, int site) {
                return mbar_wait_warp(bar(b), parity, prm.err, site, abort_flag);
            };
            if (warp == 9) {
                constexpr uint32_t idS = umma_idesc_bf16(128, kQT, false);
                const uint64_t dK = umma_desc_sw128(smem_u32(sk), 16, 1024);
                bool ok = wait_w(B_KV, 0, 60);
                for (int u = 0; ok && u < nu; ++u) {
                    const int s = u % kStages;
                    const uint32_t b = (uint32_t)(u & 1) * 64;
                    ok = wait_w(B_QFULL + s, (u / kStages) & 1, 61) && (u < 2 || wait_w(B_ACC + (u & 1), ((u >> 1) - 1) & 1, 63));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dq = umma_desc_sw128(smem_u32(sq + s * kQTile), 16, 1024);
                    umma_bf16_ss_k128_warp<1, kKPanel, kQPanel>(tmem + kColS + b, dK, dq, idS);
                    umma_commit_warp(bar(B_SFULL + (u & 1)));
                }
            } else if (warp == 11) {
                constexpr uint32_t idS = umma_idesc_bf16(128, kQT, false);
                bool ok = wait_w(B_VT, 0, 66);
                for (int u = 0; ok && u < nu; ++u) {
                    const int s = u % kStages;
                    ok = wait_w(B_QFULL + s, (u / kStages) & 1, 67) && (u == 0 || wait_w(B_DPFREE, (u - 1) & 1, 65));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dg = umma_desc_sw128(smem_u32(sg + s * kQTile), 16, 1024);
                    umma_bf16_ts_k128_warp<kQPanel>(tmem + kColDP, tmem + kColV, dg, idS);
                    umma_commit_warp(bar(B_SFULL + (u & 1)));
                }
            } else {
                constexpr uint32_t idAcc = umma_idesc_bf16(128, kD, true);
                bool ok = true;
                for (int u = 0; ok && u < nu; ++u) {
                    const int s = u % kStages;
                    const uint32_t b = (uint32_t)(u & 1) * 64;
                    if (!(ok = wait_w(B_PFULL + (u & 1), (u >> 1) & 1, 62))) break;
                    tc_fence_after();
                    // the step's Q and dO as MN-major B operands (N = head dim, K = the 64 queries)
                    const uint64_t gmn = umma_desc_sw128(smem_u32(sg + s * kQTile), kQPanel, 1024);
                    const uint64_t qmn = umma_desc_sw128(smem_u32(sq + s * kQTile), kQPanel, 1024);
                    umma_bf16_ts_k64_mn_warp<1, slice_col<kQT>(1), slice_col<kQT>(2), slice_col<kQT>(3)>(
                        tmem + kColAcc0, tmem + kColS + b, gmn, idAcc, u > 0);
                    umma_bf16_ts_k64_mn_warp<1, slice_col<kQT>(1), slice_col<kQT>(2), slice_col<kQT>(3)>(
                        tmem + kColAcc1, tmem + kColS + b + 16, qmn, idAcc, u > 0);
                    umma_commit_warp(bar(B_ACC + (u & 1)));
                    umma_commit_warp(bar(B_QEMPTY + s));
                }
            }
            // every MMA issued above must complete before tensor memory is read or released
            umma_commit_warp(bar(B_FINAL + warp - 9));
            mbar_wait_bounded(bar(B_FINAL + warp - 9), 0, prm.err, 64);
        }
    } else {
        // ---------------------------------------------------------------- softmax + epilogue
        const float c = prm.scale_log2;
        auto wait_all = [&](int b, uint32_t parity, int site) {
            return mbar_wait_warp(bar(b), parity, prm.err, site, abort_flag);
        };
        bool ok = true;
        if (nu > 0 && (ok = wait_all(B_KV, 0, 73))) {   // V's rows into tensor memory, 64 dims a thread
            uint32_t w[32];
            const uint8_t *row = sv + ch * kKPanel + (lq * 32 + lane) * 128;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint4 x = *reinterpret_cast<const uint4 *>(row + ((i ^ (lane & 7)) * 16));
                w[4 * i] = x.x; w[4 * i + 1] = x.y; w[4 * i + 2] = x.z; w[4 * i + 3] = x.w;
            }
            tmem_st32(tmem + lanes + kColV + 32 * ch, w);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            mbar_arrive_warp(bar(B_VT));
        }
        // the next step's entry, read a step ahead
        int e = e0 + ub / group, left = group - ub % group;   // steps left of entry e
        int kind = nu > 0 ? prm.kind[e] : 0, qtile = nu > 0 ? prm.idx[e] : 0;
        for (int u = 0; ok && u < nu; ++u) {
            const int s = u % kStages;
            const uint32_t b = (uint32_t)(u & 1) * 64 + 32 * ch;
            const bool partial = __any_sync(0xffffffffu, kind != PADOC_TILE_FULL);
            const int qbase = qtile * kQT + 32 * ch;
            if (!wait_all(B_QFULL + s, (u / kStages) & 1, 71) || !wait_all(B_SFULL + (u & 1), (u >> 1) & 1, 70)) {
                ok = false;
                break;
            }
            tc_fence_after();
            if (--left == 0 && u + 1 < nu) {
                left = group;
                kind = prm.kind[++e];
                qtile = prm.idx[e];
            }
            uint32_t sr[32], dr[32];
            tmem_ld32(tmem + lanes + kColS + b, sr);
            tmem_ld32(tmem + lanes + kColDP + 32 * ch, dr);
            const float4 *la = reinterpret_cast<const float4 *>(aux + s * kAuxBytes) + 8 * ch;
            const float4 *da = reinterpret_cast<const float4 *>(aux + s * kAuxBytes + kQT * 4) + 8 * ch;
            const int4 *sp = reinterpret_cast<const int4 *>(aux + s * kAuxBytes + 2 * kQT * 4) + 32 * ch;
            uint32_t vis = 0xffffffffu;
            if (partial) {   // (warp-uniform)
                // lane i: which of the warp's 32 keys query qbase + i sees (its two spans as bit
                // intervals); a 32 x 32 bit transpose across the warp then gives each key's bits over
                // the 32 queries
                const int64_t rem = prm.T - qbase;   // query columns past T hold no spans
                const int nvalid = rem <= 0 ? 0 : (rem >= 32 ? 32 : (int)rem);
                const int kbase = kt * kKT + lq * 32;
                uint32_t x = 0u;
                if (lane < nvalid) {
                    const int4 w = sp[lane];
                    const int lo0 = clamp_w(w.x - kbase, 32), lo1 = clamp_w(w.z - kbase, 32);
                    x = interval_bits(lo0, max(clamp_w(w.y - kbase, 32) - lo0, 0), 0) |
                        interval_bits(lo1, max(clamp_w(w.w - kbase, 32) - lo1, 0), 0);
                }
                vis = transpose32_warp(x, lane);
            }
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            mbar_arrive_warp(bar(B_DPFREE));
            uint32_t pk[16], dk[16];
            const uint64_t c2 = f2_pack(c, c);
            // two query columns per packed instruction: P = exp2(S c - lse2), dS = P (dP - D)
            auto column_pairs = [&](auto masked) {
#pragma unroll
                for (int i4 = 0; i4 < 8; ++i4) {
                    const float4 l4 = la[i4], d4 = da[i4];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int i = 4 * i4 + 2 * j;
                        float x0, x1;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sr[i]), __uint_as_float(sr[i + 1])), c2,
                                         j ? f2_pack(l4.z, l4.w) : f2_pack(l4.x, l4.y)), x0, x1);
                        float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                        if (decltype(masked)::value) {
                            p0 = (vis >> i) & 1u ? p0 : 0.f;
                            p1 = (vis >> (i + 1)) & 1u ? p1 : 0.f;
                        }
                        const uint64_t t = f2_sub(f2_pack(__uint_as_float(dr[i]), __uint_as_float(dr[i + 1])),
                                                  j ? f2_pack(d4.z, d4.w) : f2_pack(d4.x, d4.y));
                        float d0, d1;
                        f2_unpack(f2_mul(f2_pack(p0, p1), t), d0, d1);
                        pk[i >> 1] = pack_bf16x2(p0, p1);
                        dk[i >> 1] = pack_bf16x2(d0, d1);
                    }
                }
            };
            if (partial) column_pairs(std::true_type{}); else column_pairs(std::false_type{});
            tmem_st16(tmem + lanes + kColS + b, pk);
            tmem_st16(tmem + lanes + kColS + b + 16, dk);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            mbar_arrive_warp(bar(B_PFULL + (u & 1)));
        }
        sums = ok && (nu == 0 || wait_all(B_FINAL + 1, 0, 72));
        tc_fence_after();
    }
    // Epilogue. The 256 columns of dV | dK are split over the cluster's CTAs: each one's softmax threads
    // (a key row and half of the columns each) send the other CTAs' parts to their shared memory, which
    // nothing else uses any more, add what they receive to their own part in rank order and write it.
    constexpr int kPart = 256 / NC, kHalfPart = kPart / 2;   // columns of a CTA, of a thread
    auto part = [&](int p, int c, uint32_t (&o)[16]) {       // 16 of this CTA's sums of part p
        if (nu > 0) {
            tmem_ld16(tmem + lanes + kColAcc0 + kPart * p + kHalfPart * ch + c, o);
            tmem_ld_wait();
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = 0u;
        }
    };
    // the place of a thread's 16 columns from CTA `from` in the receiver's shared memory
    auto slot = [&](int from, int to, int c) {
        const int n = from < to ? from : from - 1;
        return (uint32_t)(n * kPart * kKT * 4 + (kHalfPart * ch + c) * kKT * 4 + (lq * 32 + lane) * 16);
    };
    if (NC > 1) {
        tc_fence_before();
        cluster_sync();
        if (sums) {
            tc_fence_after();
#pragma unroll 1
            for (int d = 1; d < NC; ++d) {
                const int p = (rank + d) % NC;
                const uint32_t dst = cluster_map(smem_u32(smem), p);
#pragma unroll 1
                for (int c = 0; c < kHalfPart; c += 16) {
                    uint32_t o[16];
                    part(p, c, o);
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        st_cluster_v4(dst + slot(rank, p, c + i), make_int4(o[i], o[i + 1], o[i + 2], o[i + 3]));
                }
            }
        }
        cluster_sync();
    }
    if (sums) {
#pragma unroll 1
        for (int c = 0; c < kHalfPart; c += 16) {
            uint32_t own[16];
            part(rank, c, own);
            float acc[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[i] = 0.f;
#pragma unroll
            for (int from = 0; from < NC; ++from)
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                    const float4 x = from == rank ? make_float4(__uint_as_float(own[i]), __uint_as_float(own[i + 1]),
                                                                __uint_as_float(own[i + 2]), __uint_as_float(own[i + 3]))
                                                  : *reinterpret_cast<const float4 *>(smem + slot(from, rank, c + i));
                    acc[i] += x.x;
                    acc[i + 1] += x.y;
                    acc[i + 2] += x.z;
                    acc[i + 3] += x.w;
                }
            const int col = kPart * rank + kHalfPart * ch + c;
            const bool isk = col >= kD;                       // dV first, then dK (times scale)
            if (key < prm.T)
                store_row_bf16((isk ? prm.out0 : prm.out1) + ((size_t)key * hkv + g) * kD + (col & (kD - 1)), acc,
                               isk ? prm.scale : 1.f);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ================================================================================================
// dQ pass
// ================================================================================================
namespace dqp {
constexpr int kQT = PADOC_BWD_DQ_Q_TILE;     // 128 query rows: the M of every MMA
constexpr int kW = PADOC_BWD_DQ_K_TILE;      // 64 keys per step
constexpr int kStages = 4;
constexpr int kQPanel = kQT * 128;           // [128 rows][64 bf16]
constexpr int kQTile = 2 * kQPanel;
constexpr int kKPanel = kW * 128;            // [64 rows][64 bf16]
constexpr int kKTile = 2 * kKPanel;          // K or V of one step
constexpr int kSlots = 3;                    // S buffers; a step's dS takes its S's place
constexpr uint32_t kColQ = 0, kColS = 64, kColDP = 256, kColDQ = 384;   // Q (A operand), S x 3, dP x 2, dQ
static_assert(kW == 64, "the accumulating block takes four K-steps");
enum {
    B_QROWS = 0,                   // the unit's Q has landed
    B_GROWS = 1,                   // its dO and O have landed
    B_QT = 2,                      // its Q is in tensor memory (an arrival per softmax warp)
    B_D = 3,                       // its rows' halves of D are in shared memory (an arrival per softmax warp)
    B_DREAD = 4,                   // ... and have been read, as dO and O (an arrival per softmax warp)
    B_QFREE = 5,                   // Q's place is free for the next unit's (an arrival per softmax warp)
    B_GFREE = 6,                   // the unit's last dP is done
    B_DQFULL = 7,                  // the unit's dQ is complete
    B_DQFREE = 8,                  // ... and read (an arrival per softmax warp)
    B_NEXT = 9,                    // the launch control's answer
    B_UFULL = 10,                  // [unit parity]
    B_UEMPTY = 12,                 // [unit parity], an arrival per reading warp
    B_KFULL = 14,                  // [stage]
    B_KEMPTY = 14 + kStages,       // [stage]
    B_SFULL = 14 + 2 * kStages,    // [slot]: S and dP (an arrival each)
    B_PFULL = 17 + 2 * kStages,    // [slot]: dS (an arrival per softmax warp)
    B_ACC = 20 + 2 * kStages,      // [slot]: the accumulating MMAs that read it are done
    B_DPFREE = 23 + 2 * kStages,   // [step parity]: dP is read (an arrival per softmax warp)
    B_FINAL = 25 + 2 * kStages,    // [issuing warp]
    B_COUNT = 28 + 2 * kStages
};
struct Unit {   // nu < 0: no more units
    int h, qt, e0, nu;
};
constexpr int kReaders = 11;       // softmax and issuing warps
constexpr size_t kSmemBytes = 1024 + 3 * (size_t)kQTile + 2 * (size_t)kStages * kKTile + B_COUNT * 8 + 2 * sizeof(Unit) + 48 +
                              2 * kQT * 4;
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
}  // namespace dqp

__global__ void __launch_bounds__(kThreads, 1)
prefill_bwd_dq_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap gmap,
                      const __grid_constant__ CUtensorMap omap, const __grid_constant__ CUtensorMap kmap,
                      const __grid_constant__ CUtensorMap vmap, const __grid_constant__ CUtensorMap dqmap,
                      const BwdParams prm)
{
    using namespace dqp;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sq = smem;                        // Q, dO and O rows; dQ leaves by way of Q's place
    uint8_t *sg = sq + kQTile;
    uint8_t *so = sg + kQTile;
    uint8_t *sk = so + kQTile;                 // [stage] K step tiles
    uint8_t *sv = sk + kStages * kKTile;       // [stage] V step tiles
    Unit *units = (Unit *)(sv + kStages * kKTile);   // [2]
    uint8_t *answer = (uint8_t *)(units + 2);  // 16 bytes
    uint64_t *bars = (uint64_t *)(answer + 16);
    uint32_t *tmem_slot = (uint32_t *)(bars + B_COUNT);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    float *dsum = (float *)(tmem_slot + 8);    // [2][128]: the two column halves' parts of D

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (a value the compiler knows to be warp-uniform)
    const int hq = prm.num_q_heads, group = hq / prm.num_kv_heads;
    pdl_launch_dependents();   // the dK/dV pass may take the SMs that run out of work here
    auto bar = [&](int i) { return smem_u32(&bars[i]); };

    if (tid == 0) {
        for (int i = 0; i < B_COUNT; ++i) {
            const bool soft = i == B_QT || i == B_D || i == B_DREAD || i == B_QFREE || i == B_DQFREE ||
                              (i >= B_PFULL && i < B_PFULL + kSlots) || i == B_DPFREE || i == B_DPFREE + 1;
            mbar_init(bar(i), soft ? 8 : i == B_UEMPTY || i == B_UEMPTY + 1 ? kReaders : i >= B_SFULL && i < B_SFULL + kSlots ? 2 : 1);
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 9) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    auto wait_w = [&](int b, uint32_t parity, int site) {
        return mbar_wait_warp(bar(b), parity, prm.err, site, abort_flag);
    };
    // the n-th unit, as every lane of a reading warp sees it
    auto read_unit = [&](int n, Unit &u, int site) {
        if (!wait_w(B_UFULL + (n & 1), (n >> 1) & 1, site)) return false;
        const Unit v = units[n & 1];
        u.h = __shfl_sync(0xffffffffu, v.h, 0);
        u.qt = __shfl_sync(0xffffffffu, v.qt, 0);
        u.e0 = __shfl_sync(0xffffffffu, v.e0, 0);
        u.nu = __shfl_sync(0xffffffffu, v.nu, 0);
        __syncwarp();   // (every lane's read has returned before the slot may be written again)
        mbar_arrive_warp(bar(B_UEMPTY + (n & 1)));
        return true;
    };

    if (warp == 8) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            auto wait = [&](int b, uint32_t parity, int site) {
                return wait_or_abort(bar(b), parity, prm.err, site, abort_flag);
            };
            int x = blockIdx.x, y = 0;
            int tk = 0, nq = 0, ng = 0;   // K/V tiles, Q tiles, dO and O tiles issued so far
            bool ok = true, more = true, asked = false;
            // asked with the unit's last tile: early enough for the answer, and late enough that no CTA
            // holds a second unit while others run out of work
            auto ask = [&]() {
                mbar_arrive_expect_tx(bar(B_NEXT), 16);
                launch_control_ask(smem_u32(answer), bar(B_NEXT));
                asked = true;
            };
            int n = 0;
            for (;; ++n) {
                if (n >= 2 && !wait(B_UEMPTY + (n & 1), ((n >> 1) - 1) & 1, 83)) break;
                Unit u = {0, 0, 0, -1};
                if (more) {
                    u.h = x % hq;
                    u.qt = prm.num_tiles - 1 - x / hq;   // heavier q-tiles (later in a page) first
                    u.e0 = prm.ptr[u.qt];
                    u.nu = max(prm.ptr[u.qt + 1] - u.e0, 0);
                }
                units[n & 1] = u;
                mbar_arrive(bar(B_UFULL + (n & 1)));
                if (u.nu < 0) break;
                if (n > 0 && !wait(B_QFREE, (n - 1) & 1, 84)) break;
                mbar_arrive_expect_tx(bar(B_QROWS), kQTile);
                for (int p = 0; p < 2; ++p)
                    tma_load_2d(smem_u32(sq) + p * kQPanel, &qmap, u.h * kD + 64 * p, u.qt * kQT, bar(B_QROWS));
                ++nq;
                // the first K and V tiles go before dO, whose place is free later
                auto load_rows = [&]() {
                    if (n > 0 && (!wait(B_DREAD, (n - 1) & 1, 85) || !wait(B_GFREE, (n - 1) & 1, 86))) return false;
                    mbar_arrive_expect_tx(bar(B_GROWS), 2 * kQTile);
                    for (int p = 0; p < 2; ++p) {
                        tma_load_2d(smem_u32(sg) + p * kQPanel, &gmap, u.h * kD + 64 * p, u.qt * kQT, bar(B_GROWS));
                        tma_load_2d(smem_u32(so) + p * kQPanel, &omap, u.h * kD + 64 * p, u.qt * kQT, bar(B_GROWS));
                    }
                    ++ng;
                    return true;
                };
                const int g = u.h / group;
                for (int j = 0; j < u.nu; ++j, ++tk) {
                    if (j + 1 == u.nu) ask();
                    const int s = tk % kStages;
                    if (tk >= kStages && !(ok = wait(B_KEMPTY + s, (tk / kStages - 1) & 1, 80))) break;
                    const int k0 = prm.idx[u.e0 + j] * kW;
                    const uint32_t fb = bar(B_KFULL + s);
                    const uint32_t kb = smem_u32(sk + s * kKTile), vb = smem_u32(sv + s * kKTile);
                    mbar_arrive_expect_tx(fb, 2 * kKTile);
                    tma_load_2d(kb, &kmap, g * kD, k0, fb);
                    tma_load_2d(kb + kKPanel, &kmap, g * kD + 64, k0, fb);
                    tma_load_2d(vb, &vmap, g * kD, k0, fb);
                    tma_load_2d(vb + kKPanel, &vmap, g * kD + 64, k0, fb);
                    if (j == 0 && !(ok = load_rows())) { ++tk; break; }
                }
                if (!ok) break;
                if (u.nu == 0) {
                    ask();
                    if (!load_rows()) break;
                }
                if (!wait(B_NEXT, n & 1, 87)) break;
                asked = false;
                more = launch_control_answer(smem_u32(answer), x, y);
                fence_proxy_async_smem();   // the answer is read before the next one may be written
            }
            // copies still in flight must land before the CTA's shared memory is released
            if (asked) mbar_wait_bounded(bar(B_NEXT), n & 1, prm.err, 88);
            if (nq) mbar_wait_bounded(bar(B_QROWS), (nq - 1) & 1, prm.err, 81);
            if (ng) mbar_wait_bounded(bar(B_GROWS), (ng - 1) & 1, prm.err, 81);
            for (int i = max(tk - kStages, 0); i < tk; ++i)
                mbar_wait_bounded(bar(B_KFULL + i % kStages), (i / kStages) & 1, prm.err, 82);
        }
    } else if (warp >= 9) {
        // ---------------------------------------------------------------- MMA issuers (whole warps)
        // warp 9 S, warp 11 dP, warp 10 dQ, as in the dK/dV pass; c counts the steps of all units
        int c = 0, slot = 0;
        uint32_t ph = 0;   // parity of the slot's use
        bool ok = true;
        auto next_step = [&]() {
            ++c;
            if (++slot == kSlots) { slot = 0; ph ^= 1; }
        };
        Unit un;
        for (int n = 0; ok && (ok = read_unit(n, un, 101)) && un.nu >= 0; ++n) {
            if (warp == 9) {
                // S = Q K^T, A from tensor memory
                constexpr uint32_t idS = umma_idesc_bf16(128, kW, false);
                ok = wait_w(B_QT, n & 1, 90);
                for (int u = 0; ok && u < un.nu; ++u, next_step()) {
                    const int s = c % kStages;
                    ok = wait_w(B_KFULL + s, (c / kStages) & 1, 91) && (c < kSlots || wait_w(B_ACC + slot, ph ^ 1, 93));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dk = umma_desc_sw128(smem_u32(sk + s * kKTile), 16, 1024);
                    umma_bf16_ts_k128_warp<kKPanel>(tmem + kColS + 64 * slot, tmem + kColQ, dk, idS);
                    umma_commit_warp(bar(B_SFULL + slot));
                }
            } else if (warp == 11) {
                // dP = dO V^T, both from shared memory
                constexpr uint32_t idS = umma_idesc_bf16(128, kW, false);
                const uint64_t dg = umma_desc_sw128(smem_u32(sg), 16, 1024);
                ok = wait_w(B_GROWS, n & 1, 97);
                for (int u = 0; ok && u < un.nu; ++u, next_step()) {
                    const int s = c % kStages;
                    ok = wait_w(B_KFULL + s, (c / kStages) & 1, 98) &&
                         (c < 2 || wait_w(B_DPFREE + (c & 1), ((c >> 1) - 1) & 1, 99));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t dv = umma_desc_sw128(smem_u32(sv + s * kKTile), 16, 1024);
                    umma_bf16_ss_k128_warp<1, kQPanel, kKPanel>(tmem + kColDP + 64 * (c & 1), dg, dv, idS);
                    umma_commit_warp(bar(B_SFULL + slot));
                }
                umma_commit_warp(bar(B_GFREE));
            } else {
                constexpr uint32_t idAcc = umma_idesc_bf16(128, kD, true);
                for (int u = 0; ok && u < un.nu; ++u, next_step()) {
                    const int s = c % kStages;
                    // (the dQ of the unit before is read before this one's first product overwrites it)
                    ok = wait_w(B_PFULL + slot, ph, 92) && (u > 0 || n == 0 || wait_w(B_DQFREE, (n - 1) & 1, 102));
                    if (!ok) break;
                    tc_fence_after();
                    // the step's K as an MN-major B operand (N = head dim, K = the 64 keys)
                    const uint64_t kmn = umma_desc_sw128(smem_u32(sk + s * kKTile), kKPanel, 1024);
                    umma_bf16_ts_k64_mn_warp<1, slice_col<kW>(1), slice_col<kW>(2), slice_col<kW>(3)>(
                        tmem + kColDQ, tmem + kColS + 64 * slot, kmn, idAcc, u > 0);
                    umma_commit_warp(bar(B_ACC + slot));
                    umma_commit_warp(bar(B_KEMPTY + s));
                }
                // A unit without entries issued nothing above and waited for nothing: its commit would complete the
                // phase right behind the unit before's, whose parity the softmax warps may not have seen yet.
                if (ok && un.nu == 0 && n > 0) ok = wait_w(B_DQFREE, (n - 1) & 1, 102);
                umma_commit_warp(bar(B_DQFULL));
            }
        }
        umma_commit_warp(bar(B_FINAL + warp - 9));
        mbar_wait_bounded(bar(B_FINAL + warp - 9), 0, prm.err, 94);
    } else {
        // ---------------------------------------------------------------- softmax + epilogue
        const int lq = warp & 3, ch = warp >> 2;
        const int row = lq * 32 + lane;
        const uint32_t lanes = (uint32_t)(lq * 32) << 16;
        const uint64_t c2 = f2_pack(prm.scale_log2, prm.scale_log2);
        uint8_t *qrow = sq + ch * kQPanel + row * 128;
        const uint8_t *grow = sg + ch * kQPanel + row * 128, *orow = so + ch * kQPanel + row * 128;
        int c = 0, slot = 0;   // steps of all units
        uint32_t ph = 0;
        Unit un, last = {0, 0, 0, 0};
        bool ok = true;
        for (int n = 0; ok && (ok = read_unit(n, un, 103)); ++n) {
            const int64_t t = (int64_t)un.qt * kQT + row;
            const bool in = un.nu >= 0 && t < prm.T;
            int a0 = 0, a1 = 0, b0 = 0, b1 = 0, kind = 0, ktile = 0;   // kind, ktile: the next step's entry
            float nlrow = -INFINITY;
            if (un.nu >= 0) {
                if (in) {
                    const int4 w = *reinterpret_cast<const int4 *>(prm.spans + 4 * t);
                    a0 = w.x; a1 = w.y; b0 = w.z; b1 = w.w;
                    const float l = prm.lse[(size_t)t * hq + un.h];
                    nlrow = l == -INFINITY ? -INFINITY : -l * PADOC_LOG2E;
                }
                if (un.nu > 0) {
                    kind = prm.kind[un.e0];
                    ktile = prm.idx[un.e0];
                }
                // Q's row of this query into tensor memory (dims 64 ch .. 64 ch + 63); the S of the unit before
                // that read the last one are done, as their steps are
                if (!(ok = wait_w(B_QROWS, n & 1, 100))) break;
                uint32_t w[32];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(qrow + ((i ^ (lane & 7)) * 16));
                    w[4 * i] = x.x; w[4 * i + 1] = x.y; w[4 * i + 2] = x.z; w[4 * i + 3] = x.w;
                }
                tmem_st32(tmem + lanes + kColQ + 32 * ch, w);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                mbar_arrive_warp(bar(B_QT));
            }
            // the unit before's dQ times scale, columns 64 ch .. 64 ch + 63 of the thread's row, by way of this
            // warp's part of Q's place and one TMA store per warp, which leaves out the rows past T
            if (n > 0) {
                if (!(ok = wait_w(B_DQFULL, (n - 1) & 1, 96))) break;
                tc_fence_after();
                uint32_t o[2][32];
                if (last.nu > 0) {
                    tmem_ld32(tmem + lanes + kColDQ + 64 * ch, o[0]);
                    tmem_ld32(tmem + lanes + kColDQ + 64 * ch + 32, o[1]);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[0][i] = o[1][i] = 0u;
                }
                tc_fence_before();
                __syncwarp();
                mbar_arrive_warp(bar(B_DQFREE));
#pragma unroll
                for (int i = 0; i < 64; i += 8) {
                    auto v = [&](int k) { return __uint_as_float(o[i >> 5][(i & 31) + k]) * prm.scale; };
                    *reinterpret_cast<uint4 *>(qrow + (((i / 8) ^ (lane & 7)) * 16)) =
                        make_uint4(pack_bf16x2(v(0), v(1)), pack_bf16x2(v(2), v(3)), pack_bf16x2(v(4), v(5)), pack_bf16x2(v(6), v(7)));
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&dqmap, last.h * kD + 64 * ch, last.qt * kQT + lq * 32, smem_u32(sq + ch * kQPanel + lq * 4096));
                    tma_store_commit();
                    tma_store_wait_read<0>();   // before the next unit's Q, or the release of shared memory
                }
                __syncwarp();
            }
            if (un.nu < 0) break;
            if (lane == 0) mbar_arrive(bar(B_QFREE));
            last = un;
            // the row's statistics: D = dO . O (fp32, the two column halves added through shared memory)
            // and -lse2; rows past T (zeros in the tiles) get -lse2 = -inf and D = 0, so that their P and dS
            // are 0. Every (row, head) of [0, t_pad) belongs to exactly one unit, which writes them for the
            // dK/dV pass.
            if (!(ok = wait_w(B_GROWS, n & 1, 104) && (n == 0 || wait_w(B_DREAD, (n - 1) & 1, 105)))) break;
            uint64_t acc2 = f2_pack(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint4 x = *reinterpret_cast<const uint4 *>(grow + ((i ^ (lane & 7)) * 16));
                const uint4 y = *reinterpret_cast<const uint4 *>(orow + ((i ^ (lane & 7)) * 16));
                const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc2 = f2_fma(f2_pack(__uint_as_float(xs[j] << 16), __uint_as_float(xs[j] & 0xffff0000u)),
                                  f2_pack(__uint_as_float(ys[j] << 16), __uint_as_float(ys[j] & 0xffff0000u)), acc2);
            }
            float lo, hi;
            f2_unpack(acc2, lo, hi);
            dsum[ch * kQT + row] = lo + hi;
            __syncwarp();
            mbar_arrive_warp(bar(B_D));
            if (!(ok = wait_w(B_D, n & 1, 106))) break;
            const float drow = in ? dsum[row] + dsum[kQT + row] : 0.f;
            __syncwarp();
            mbar_arrive_warp(bar(B_DREAD));
            if (ch == 0) {
                prm.lt[(size_t)un.h * prm.t_pad + t] = nlrow;
                prm.dt[(size_t)un.h * prm.t_pad + t] = drow;
            }
            const uint64_t nl2 = f2_pack(nlrow, nlrow), d2 = f2_pack(drow, drow);
            for (int u = 0; ok && u < un.nu; ++u, ++c) {
                const uint32_t b = tmem + lanes + kColS + 64 * slot + 32 * ch;
                const bool partial = __any_sync(0xffffffffu, kind != PADOC_TILE_FULL);
                const int cb = ktile * kW + 32 * ch;
                if (!(ok = wait_w(B_SFULL + slot, ph, 95))) break;
                tc_fence_after();
                if (u + 1 < un.nu) {
                    kind = prm.kind[un.e0 + u + 1];
                    ktile = prm.idx[un.e0 + u + 1];
                }
                uint32_t sr[32], dr[32];
                tmem_ld32(b, sr);
                tmem_ld32(tmem + lanes + kColDP + 64 * (c & 1) + 32 * ch, dr);
                uint32_t vis = 0xffffffffu;
                if (partial) {
                    const int lo0 = clamp_w(a0 - cb, 32), lo1 = clamp_w(b0 - cb, 32);
                    vis = interval_bits(lo0, max(clamp_w(a1 - cb, 32) - lo0, 0), 0) |
                          interval_bits(lo1, max(clamp_w(b1 - cb, 32) - lo1, 0), 0);
                }
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                mbar_arrive_warp(bar(B_DPFREE + (c & 1)));
                uint32_t dk[16];
                // two key columns per packed instruction: P = exp2(S c - lse2), dS = P (dP - D)
                auto column_pairs = [&](auto masked) {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        float x0, x1;
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(sr[i]), __uint_as_float(sr[i + 1])), c2, nl2), x0, x1);
                        float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                        if (decltype(masked)::value) {
                            p0 = (vis >> i) & 1u ? p0 : 0.f;
                            p1 = (vis >> (i + 1)) & 1u ? p1 : 0.f;
                        }
                        const uint64_t t2 = f2_sub(f2_pack(__uint_as_float(dr[i]), __uint_as_float(dr[i + 1])), d2);
                        float d0, d1;
                        f2_unpack(f2_mul(f2_pack(p0, p1), t2), d0, d1);
                        dk[i >> 1] = pack_bf16x2(d0, d1);
                    }
                };
                if (partial) column_pairs(std::true_type{}); else column_pairs(std::false_type{});
                tmem_st16(b, dk);   // over the first half of this thread's own S columns
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                mbar_arrive_warp(bar(B_PFULL + slot));
                if (++slot == kSlots) { slot = 0; ph ^= 1; }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// The CTAs that share a dK/dV unit. A page's first k-tiles are seen by all of its later queries, so the
// largest unit is about twice the mean and a few units leave most of the chip idle; with many units, or units
// of few steps, the sharing's own cost (~8 us a CTA) is the larger. The host knows the number of units, the
// query heads of a KV head (`group`: a unit's steps per q-tile) and a bound on the steps (every q-tile of the
// call), not the page lengths, so the lines suit batches of short pages too. Measured on 152 SMs over 258
// calls (13 head shapes, 40 to 20k tokens, pages of 60 to 6000), both passes, with 1 / 2 / 4 / 8 CTAs a unit:
//   group 8: one page of 3419 tokens (54 units) 368 / 215 / 137 / 156 us, 34107 packed tokens (534 units)
//            1179 / 1159 / 1249 / 1517 us, 40 pages of 60 tokens (38 units) 40 / 29 / 34 / 44 us;
//   group 4: 16 pages of 140 tokens (144 units) 47 / 49 / 66 / 121 us, one page of 2500 tokens (80) 152 / 96 / 83 / 119 us;
//   group 1: 8 pages of 140 tokens (144 units) 18.9 / 27 / 44 / 99 us, one page of 2500 tokens (20) 52 / 39 / 32 / 35 us.
// On none of the 258 calls is the choice slower (by more than the spread) than the kernel before the clusters.
int pick_cluster(int64_t units, int group, int64_t total_tokens)
{
    const int64_t u = units * 152 / padoc_default_ctas(), steps = (total_tokens + dkv::kQT - 1) / dkv::kQT * group;
    if (group >= 6) return u <= 45 ? 8 : u <= 160 ? 4 : u <= 560 ? 2 : 1;
    int nc;
    if (group >= 3) nc = u <= 12 ? 8 : u <= (steps >= 280 ? 160 : 72) ? 4 : u <= 560 ? 2 : 1;
    else nc = u <= 12 ? 8 : u <= 36 ? 4 : u <= (steps >= 40 ? 100 : 76) ? 2 : 1;
    while (nc > 1 && nc >= steps) nc /= 2;   // a step or more for each
    return nc;
}

template <int NC>
padoc_status launch_dkv(const CUtensorMap &q64, const CUtensorMap &g64, const CUtensorMap &k128, const CUtensorMap &v128,
                        const BwdParams &prm, int64_t units, cudaStream_t stream)
{
    auto kernel = prefill_bwd_dkv_kernel<NC>;
    if (const padoc_status st = padoc_set_max_smem((const void *)kernel, (int)dkv::kSmemBytes)) return st;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(units * NC));
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = dkv::kSmemBytes;
    lc.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = NC;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see the producer's wait
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 2;
    PADOC_CUDA_TRY(cudaLaunchKernelEx(&lc, kernel, q64, g64, k128, v128, prm));
    return padoc_launch_status();
}

}  // namespace

padoc_status padoc_launch_prefill_bwd_tc(const void *q, const void *k, const void *v, const void *out,
                                         const void *dout, const float *lse, int64_t total_tokens,
                                         int32_t num_q_heads, int32_t num_kv_heads, const int32_t *spans_dev,
                                         const padoc_tile_map_dev *q_map, const padoc_tile_map_dev *k_map, float *lt,
                                         float *dt, int64_t t_pad, float scale, void *dq, void *dk,
                                         void *dv, cudaStream_t stream)
{
    int *err = padoc_device_error_word();
    if (!err) return PADOC_ERR_CUDA;
    const int64_t T = total_tokens;
    const int64_t nkt = (T + dkv::kKT - 1) / dkv::kKT, nqt = (T + dqp::kQT - 1) / dqp::kQT;
    if (2 * nkt * num_kv_heads > INT32_MAX || nqt * num_q_heads > INT32_MAX) return PADOC_ERR_UNSUPPORTED;   // (8 CTAs a unit: few units)
    const uint64_t qcols = (uint64_t)num_q_heads * kD, kcols = (uint64_t)num_kv_heads * kD;
    CUtensorMap q64, g64, k128, v128, k64, v64, q128, g128, o128, dq32;
    if (!padoc_make_tmap_bf16(&q64, q, qcols, T, qcols * 2, 64, dkv::kQT) ||
        !padoc_make_tmap_bf16(&g64, dout, qcols, T, qcols * 2, 64, dkv::kQT) ||
        !padoc_make_tmap_bf16(&k128, k, kcols, T, kcols * 2, 64, dkv::kKT) ||
        !padoc_make_tmap_bf16(&v128, v, kcols, T, kcols * 2, 64, dkv::kKT) ||
        !padoc_make_tmap_bf16(&k64, k, kcols, T, kcols * 2, 64, dqp::kW) ||
        !padoc_make_tmap_bf16(&v64, v, kcols, T, kcols * 2, 64, dqp::kW) ||
        !padoc_make_tmap_bf16(&q128, q, qcols, T, qcols * 2, 64, dqp::kQT) ||
        !padoc_make_tmap_bf16(&g128, dout, qcols, T, qcols * 2, 64, dqp::kQT) ||
        !padoc_make_tmap_bf16(&o128, out, qcols, T, qcols * 2, 64, dqp::kQT) ||
        !padoc_make_tmap_bf16(&dq32, dq, qcols, T, qcols * 2, 64, 32))
        return PADOC_ERR_CUDA;
    BwdParams prm;
    prm.spans = spans_dev;
    prm.lt = lt;
    prm.dt = dt;
    prm.T = T;
    prm.t_pad = t_pad;
    prm.num_q_heads = num_q_heads;
    prm.num_kv_heads = num_kv_heads;
    prm.scale_log2 = scale * PADOC_LOG2E;
    prm.scale = scale;
    prm.err = err;
    prm.lse = nullptr;

    // the dQ pass first: it also writes -lse2 and D of every row for the dK/dV pass
    BwdParams pq = prm;   // dQ pass over the query-major map
    pq.ptr = q_map->ptr;
    pq.idx = q_map->idx;
    pq.kind = q_map->kind;
    pq.order = nullptr;
    pq.num_tiles = (int32_t)nqt;
    pq.out0 = pq.out1 = nullptr;
    pq.lse = lse;
    if (const padoc_status sm = padoc_set_max_smem((const void *)prefill_bwd_dq_kernel, (int)dqp::kSmemBytes)) return sm;
    prefill_bwd_dq_kernel<<<(unsigned)(nqt * num_q_heads), kThreads, dqp::kSmemBytes, stream>>>(q128, g128, o128, k64, v64,
                                                                                             dq32, pq);
    padoc_status st = padoc_launch_status();
    if (st != PADOC_OK) return st;

    BwdParams pk = prm;   // dK/dV pass over the key-major map
    pk.ptr = k_map->ptr;
    pk.idx = k_map->idx;
    pk.kind = k_map->kind;
    pk.order = k_map->order;
    pk.num_tiles = (int32_t)nkt;
    pk.out0 = (__nv_bfloat16 *)dk;
    pk.out1 = (__nv_bfloat16 *)dv;
    const int64_t units = nkt * num_kv_heads;
    switch (pick_cluster(units, num_q_heads / num_kv_heads, T)) {
        case 8: return launch_dkv<8>(q64, g64, k128, v128, pk, units, stream);
        case 4: return launch_dkv<4>(q64, g64, k128, v128, pk, units, stream);
        case 2: return launch_dkv<2>(q64, g64, k128, v128, pk, units, stream);
        default: return launch_dkv<1>(q64, g64, k128, v128, pk, units, stream);
    }
}
