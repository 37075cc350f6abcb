// prefill_tc.cu -- C3 on the 5th-generation tensor cores: packed variable-length ancestor prefill
// (App. C.1: the causal problem over M and one bottom-right-aligned causal problem per branch over
// [K_{M<=f_k}; K_{Y_k}], computed in packed order without a gather).
//
// A work unit is a 128-row q-tile of four query heads sharing a KV head, run by a CTA pair (two heads
// per CTA); in small calls, and when the GQA group is no multiple of four, it is the q-tile of one head or
// of two, run by one CTA (in calls between, whichever suits the map: kEither below). It walks the q-tile's entries of the tile map: fully masked k-tiles are never
// visited, FULL tiles skip masking, PARTIAL tiles mask each row with its two spans.
//
// What bounds it and why this split (8 pages, 34107 packed tokens, 16 / 2 heads; clock64 timelines):
// - Shared-memory bandwidth. A 128 x 128 x 16 MMA with both operands in shared memory reads 8 KB in its
//   64 cycles, all that shared memory delivers. A pair's MMA (M = 256, cta_group::2) takes half of
//   B from each CTA: 96 bytes a cycle for S, 32 for P V, and half the TMA writes and L2 reads.
// - The chain softmax -> P V -> next S of one head. S, P and O of two heads fill tensor memory, so S
//   comes in halves of 64 keys in two buffers per head: the S of a half is computed while the softmax
//   works on the other half (with one 128-key S per head the softmax waited 1300 of every 3300 cycles).
// - Each wait and each MMA costs the issuing warp time (a wait behind 16 MMAs ~280 cycles, an MMA ~25),
//   so each head has its own issuing warp.
// - The ends of a unit. The grid has one CTA (pair) per unit, heavier q-tiles first, but one that runs
//   takes over pending ones' units (cluster launch control: a CTA not yet launched is cancelled and its
//   index handed over). Every SM runs one CTA for the whole call, the next unit's queries, first K/V
//   tiles and first S come under the softmax warps' output, which leaves through shared memory and the
//   TMA (16-byte stores of a row per thread cost 30 us of the call's 400).
// Together 400 -> 332 us (1.03 -> 1.25 PFLOP/s of visible entries; 338 before the waits of
// mbar_wait_warp); what is left is the tensor cores' 1152 cycles a half of both heads (of ~1450) and the
// units' ends (~4000 cycles).
//
// Warp roles (384 threads):
//   warps 0-3 / 4-7  softmax + epilogue of head 0 / head 1; thread t owns query row t (TMEM lane
//                    t), so row max and row sum need no shuffles;
//   warp 8           TMA producer: each unit's Q (per head), then K and V tiles into rings of kStages; it
//                    also asks for the next unit and announces it to the other warps (and CTA);
//   warps 9, 10      MMA issuer of head 0 / head 1 (converged warp, one elected lane; in a pair the
//                    first CTA's); warp 9 also allocates TMEM.
// TMEM (512 columns): head i keeps S_i of half h at columns 128i + 64h and O_i at 256+128i. The softmax
// writes P_i as packed bf16 over the first 32 columns of the half's S_i, and O_i += P_i V reads P_i
// straight from TMEM (V as an MN-major shared-memory operand). For a head and half the MMAs run
// S(t) -> P(t) -> PV(t) -> S(t+1) in issue order, so S(t+1) never overwrites a P still being read.
// O is rescaled lazily: the reference maximum only moves when a row's maximum grows by more than
// 2^8, which keeps every P entry <= 256 and the arithmetic exact up to rounding.
// Every wait is bounded; a wait that runs out records an error, all roles leave their loops, the
// MMA issuers wait for their MMAs, the producer for its copies, and TMEM is released.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "tc.cuh"

namespace {

constexpr int kD = 128;
constexpr int kQT = PADOC_PREFILL_Q_TILE;
constexpr int kKT = PADOC_PREFILL_K_TILE;
constexpr int kPanel = 128 * 128;    // [128 rows][64 bf16]
constexpr int kTile = 2 * kPanel;    // 32 KB
constexpr uint32_t kTmemCols = 512;
constexpr int kThreads = 384;

// NH heads per CTA, CG CTAs per unit.
template <int NH, int CG>
struct Cfg {
    static constexpr int kStages = CG == 2 ? 3 : 2;
    static constexpr int kOutPanels = CG;            // [32 rows][64 dims] of output staging per softmax warp
    static constexpr int kOutBytes = 8 * 4096 * kOutPanels;
    static constexpr int kHalf = kTile / CG;         // a CTA's part of a K or V tile
    static constexpr int kKPanel = kPanel / 2 / CG;  // 64 dims of its keys of one half
    enum {
        B_QFULL = 0,                    // [head]
        B_QEMPTY = 2,                   // [head]
        B_SFULL = 4,                    // [head][half]
        B_PFULL = 8,                    // [head][half], one arrival per warp of the head (both CTAs')
        B_PVDONE = 12,                  // [head][half]
        B_OFREE = 16,                   // [head], one arrival per warp of the head (both CTAs')
        B_UFULL = 18,                   // [slot]: the announced unit
        B_UEMPTY = 20,                  // [slot], one arrival per reading warp (both CTAs')
        B_NEXT = 22,                    // the answer of the cluster launch control
        B_FINAL = 23,                   // [head]
        B_KFULL = 25,                   // [stage]
        B_KEMPTY = B_KFULL + kStages,   // [stage], one arrival per head
        B_VFULL = B_KEMPTY + kStages,   // [stage]
        B_VEMPTY = B_VFULL + kStages,   // [stage], one arrival per head
        B_COUNT = B_VEMPTY + kStages
    };
    static constexpr int kReaders = CG == 2 ? 19 : 5 * NH;   // softmax warps, MMA warps, the second CTA's producer
    static constexpr size_t kSmemBytes = 1024 + 2 * (size_t)kTile + 2 * (size_t)kStages * kHalf + kOutBytes + 64 +
                                         B_COUNT * 8 + 64;
    static_assert(kSmemBytes <= 227 * 1024 && (CG == 1 || NH == 2), "");
};

struct TcPrefillParams {
    const int32_t *spans, *row_ptr, *tile_k;
    const int8_t *tile_kind;
    int64_t T;
    int32_t num_q_heads, num_kv_heads, num_q_tiles;
    float over;             // kEither: (q-tile, head) units an SM, less one
    float scale_log2;
    float *lse;
    int *err;
};

// A unit as the producer announces it: ne < 0 ends the CTA.
struct Unit {
    int32_t h0, qt, e0, ne;
};

// kCluster: the wait also acquires what the cluster's other CTA wrote to shared memory.
template <bool kCluster>
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, int *err, int site, volatile int *abort_flag)
{
    if (kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (kCluster ? mbar_wait_bounded_cluster(bar, parity, err, site) : mbar_wait_bounded(bar, parity, err, site)) return true;
    *abort_flag = 1;
    return false;
}

__device__ __forceinline__ int clamp_tile(int x) { return min(max(x, 0), kKT); }

constexpr int kEitherTiles = 160;   // q-tiles a kEither call may have (two units an SM, two heads and more)

// Whether a call of 1 + over (q-tile, head) units an SM is faster with one head a CTA than with two (see the
// launch). One head's longest unit takes 0.65 of the time less a tile, but the units then come in two waves:
// the second adds about 0.75 of the mean unit's tiles and a unit's start and end for its share of the SMs.
__device__ __forceinline__ bool one_head_units(int longest, int total, int q_tiles, float over)
{
    return 0.65f * (float)longest >= 2.f + over * (1.f + 0.75f * (float)total / (float)q_tiles);
}

// kEither (NH 2, one CTA): the grid has a CTA per (q-tile, head). Where the map is better run as that, only
// head 0's warps work; else the first half of the CTAs run units of two heads, and the others, past the
// units, are taken back by those that run (or end at once).
template <int NH, int CG, bool kEither = false>
__global__ void __launch_bounds__(kThreads, 1)
prefill_tc_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                  const __grid_constant__ CUtensorMap vmap, const __grid_constant__ CUtensorMap omap, const TcPrefillParams prm)
{
    using C = Cfg<NH, CG>;
    constexpr int kStages = C::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sq = smem;                       // [2 heads] tiles
    uint8_t *sk = sq + 2 * kTile;             // [kStages][key half][dim half] (CG 2: this CTA's half of the keys)
    uint8_t *sv = sk + kStages * C::kHalf;    // [kStages] tiles (CG 2: this CTA's 64 dims)
    uint8_t *so = sv + kStages * C::kHalf;    // [8 warps][kOutPanels][32][128 bytes]
    Unit *units = (Unit *)(so + C::kOutBytes);   // [2]
    uint8_t *answer = (uint8_t *)(units + 2); // 16 bytes
    uint64_t *bars = (uint64_t *)(so + C::kOutBytes + 64);
    uint32_t *tmem_slot = (uint32_t *)(bars + C::B_COUNT);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (a value the compiler knows to be warp-uniform)
    const uint32_t rank = CG == 2 ? cluster_rank() : 0;
    static_assert(!kEither || (NH == 2 && CG == 1), "");
    // the first unit's entries (for the producer), on their way while the barriers are set up: a call of one tile
    // a q-tile waits for each global read in turn
    // ([1]: as one head's unit)
    int first[kEither ? 2 : 1][2] = {};
    if (warp == 8)
#pragma unroll
        for (int k = 0; k < (kEither ? 2 : 1); ++k) {
            const int y = k ? (int)(blockIdx.y * gridDim.x + blockIdx.x) / prm.num_q_heads : (int)blockIdx.y;
            const int qt = max(prm.num_q_tiles - 1 - y, 0);   // (kEither: y past the units of two heads)
            first[k][0] = prm.row_ptr[qt];
            first[k][1] = prm.row_ptr[qt + 1];
        }
    // kEither: every warp reads the map's row pointers
    int rows[kEither ? kEitherTiles / 32 : 1][2], total = 0;
    if (kEither) {
        total = prm.row_ptr[prm.num_q_tiles];
#pragma unroll
        for (int k = 0; k < kEitherTiles / 32; ++k) {
            const int i = min(32 * k + lane, prm.num_q_tiles - 1);
            rows[k][0] = prm.row_ptr[i];
            rows[k][1] = prm.row_ptr[i + 1];
        }
    }
    auto one_head = [&]() {
        int longest = 0;
#pragma unroll
        for (int k = 0; k < kEitherTiles / 32; ++k) longest = max(longest, rows[k][1] - rows[k][0]);
        return one_head_units(__reduce_max_sync(0xffffffffu, longest), __shfl_sync(0xffffffffu, total, 0), prm.num_q_tiles, prm.over);
    };
    if constexpr (kEither)
        if ((int)blockIdx.y >= prm.num_q_tiles && !one_head()) return;
    auto bar = [&](int i) { return smem_u32(&bars[i]); };
    // a barrier of the pair's first CTA, which issues the MMAs and announces the units
    auto lead_bar = [&](int i) { return CG == 2 ? cluster_map(bar(i), 0) : bar(i); };
    auto arrive_lead = [&](int i) {
        if (CG == 2) mbar_arrive_cluster<false>(lead_bar(i));
        else mbar_arrive(bar(i));
    };

    if (tid == 0) {
        for (int i = 0; i < C::B_COUNT; ++i) {
            int n = 1;
            if (i >= C::B_PFULL && i < C::B_PFULL + 4) n = 4 * CG;
            if (i == C::B_OFREE || i == C::B_OFREE + 1) n = 4 * CG;
            if (i >= C::B_KEMPTY && i < C::B_KEMPTY + kStages) n = NH;
            if (i >= C::B_VEMPTY && i < C::B_VEMPTY + kStages) n = NH;
            if (i == C::B_UEMPTY || i == C::B_UEMPTY + 1) n = C::kReaders;
            mbar_init(bar(i), n);
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 9) {
        tmem_alloc<CG>(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish<CG>();
    }
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync();   // no arrival or copy for the other CTA before its barriers are set up
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    bool single = false;
    if constexpr (kEither) single = one_head();
    // the n-th unit, as every lane of a reading warp sees it
    auto read_unit = [&](int n, Unit &u, int site) {
        const bool r = wait_or_abort<CG == 2>(bar(C::B_UFULL + (n & 1)), (n >> 1) & 1, prm.err, site, abort_flag);
        if (!__all_sync(0xffffffffu, r)) return false;
        const Unit v = units[n & 1];
        // (every lane's read has returned before the arrival lets the slot be written again)
        u.h0 = __shfl_sync(0xffffffffu, v.h0, 0);
        u.qt = __shfl_sync(0xffffffffu, v.qt, 0);
        u.e0 = __shfl_sync(0xffffffffu, v.e0, 0);
        u.ne = __shfl_sync(0xffffffffu, v.ne, 0);
        __syncwarp();
        if (lane == 0) {
            arrive_lead(C::B_UEMPTY + (n & 1));
            if (single) arrive_lead(C::B_UEMPTY + (n & 1));   // (for head 1's warps, which have ended)
        }
        return true;
    };

    if (warp >= 8) {
        if (warp == 8 && lane == 0) {
            // ------------------------------------------------------------ TMA producer
            tma_prefetch_desc(&qmap);
            tma_prefetch_desc(&kmap);
            tma_prefetch_desc(&vmap);
            auto wait = [&](int b, uint32_t parity, int site) {
                return wait_or_abort<false>(bar(b), parity, prm.err, site, abort_flag);
            };
            // the first CTA's barrier counts both CTAs' bytes
            auto expect = [&](int b, uint32_t bytes) {
                if (rank == 0) mbar_arrive_expect_tx(bar(b), CG * bytes);
            };
            auto box = [&](uint8_t *dst, const CUtensorMap *map, int x, int y, int b) {
                if (CG == 2) tma_load_2d_pair(smem_u32(dst), map, x, y, lead_bar(b));
                else tma_load_2d(smem_u32(dst), map, x, y, bar(b));
            };
            const int group = prm.num_q_heads / prm.num_kv_heads;
            int x = blockIdx.x, y = blockIdx.y;
            int tk = 0, tv = 0, nq[2] = {0, 0};   // K and V tiles, and queries per head, issued so far
            bool ok = true, more = true, asked = false;
            // asked with the unit's last tile, a few tiles ahead of the MMAs: early enough for the answer,
            // and late enough that no CTA holds a second unit while others run out of work
            auto ask = [&]() {
                if (rank != 0) return;
                mbar_arrive_expect_tx(bar(C::B_NEXT), 16);
                launch_control_ask(smem_u32(answer), bar(C::B_NEXT));
                asked = true;
            };
            auto load_q = [&](int i, int h, int qt) {
                if (nq[i] && !wait(C::B_QEMPTY + i, (nq[i] - 1) & 1, 20)) return false;
                expect(C::B_QFULL + i, kTile);
                box(sq + i * kTile, &qmap, h * kD, qt * kQT, C::B_QFULL + i);
                box(sq + i * kTile + kPanel, &qmap, h * kD + 64, qt * kQT, C::B_QFULL + i);
                ++nq[i];
                return true;
            };
            int n = 0, asks = 0;   // units announced, questions answered
            for (;; ++n) {
                Unit u = {0, 0, 0, -1};
                if (rank == 0) {
                    if (n >= 2 && !wait(C::B_UEMPTY + (n & 1), ((n >> 1) - 1) & 1, 24)) break;
                    if (more) {
                        u.h0 = x * NH;
                        u.qt = prm.num_q_tiles - 1 - y;   // heavier tiles (later in a page) first
                        if (single) {
                            const int i = y * (int)gridDim.x + x;
                            u.h0 = i % prm.num_q_heads;
                            u.qt = prm.num_q_tiles - 1 - i / prm.num_q_heads;
                        }
                        constexpr int kOne = kEither ? 1 : 0;
                        u.e0 = n > 0 ? prm.row_ptr[u.qt] : single ? first[kOne][0] : first[0][0];
                        u.ne = (n > 0 ? prm.row_ptr[u.qt + 1] : single ? first[kOne][1] : first[0][1]) - u.e0;
                    }
                    units[n & 1] = u;
                    mbar_arrive(bar(C::B_UFULL + (n & 1)));
                    if (CG == 2) {
                        st_cluster_v4(cluster_map(smem_u32(&units[n & 1]), 1), make_int4(u.h0, u.qt, u.e0, u.ne));
                        mbar_arrive_cluster<true>(cluster_map(bar(C::B_UFULL + (n & 1)), 1));
                    }
                } else {
                    if (!wait_or_abort<true>(bar(C::B_UFULL + (n & 1)), (n >> 1) & 1, prm.err, 25, abort_flag)) break;
                    u = units[n & 1];
                }
                if (u.ne < 0) break;
                const int g = u.h0 / group, h = u.h0 + NH * (int)rank;
                int kt = u.ne > 0 ? prm.tile_k[u.e0] : 0;
                for (int j = 0; j < u.ne; ++j) {
                    if (j + 1 == u.ne) ask();
                    const int kt_next = j + 1 < u.ne ? prm.tile_k[u.e0 + j + 1] : 0;
                    // (the first K tile between the two heads' queries: S_0 needs it first)
                    if (j == 0 && !(ok = load_q(0, h, u.qt))) break;
                    const int s = tk % kStages;
                    if (tk >= kStages && !(ok = wait(C::B_KEMPTY + s, (tk / kStages - 1) & 1, 21))) break;
                    uint8_t *kb = sk + s * C::kHalf;
                    expect(C::B_KFULL + s, C::kHalf);
                    if (single) mbar_arrive(bar(C::B_KEMPTY + s));   // (for head 1, as below)
#pragma unroll
                    for (int b = 0; b < 4; ++b)   // [key half][dim half]
                        box(kb + b * C::kKPanel, &kmap, g * kD + 64 * (b & 1),
                            kt * kKT + 64 * (b >> 1) + 64 / CG * (int)rank, C::B_KFULL + s);
                    ++tk;
                    if (j == 0 && NH == 2 && !single && !(ok = load_q(1, h + 1, u.qt))) break;
                    if (tv >= kStages && !(ok = wait(C::B_VEMPTY + s, (tv / kStages - 1) & 1, 23))) break;
                    uint8_t *vb = sv + s * C::kHalf;
                    expect(C::B_VFULL + s, C::kHalf);
                    if (single) mbar_arrive(bar(C::B_VEMPTY + s));
                    box(vb, &vmap, g * kD + 64 * (int)rank, kt * kKT, C::B_VFULL + s);
                    if (CG == 1) box(vb + kPanel, &vmap, g * kD + 64, kt * kKT, C::B_VFULL + s);
                    ++tv;
                    kt = kt_next;
                }
                if (!ok) break;
                if (rank != 0) {
                    // Only now may the first CTA write this slot of ours again (it does two units on): with
                    // cluster scope, so that its stores come after the reads above, which an arrival of
                    // CTA scope straight behind them did not order. The unit's loads are issued: nothing waits.
                    mbar_arrive_cluster<true>(lead_bar(C::B_UEMPTY + (n & 1)));
                } else {
                    if (u.ne == 0) ask();
                    for (;;) {
                        if (!(ok = wait(C::B_NEXT, asks & 1, 26))) break;
                        ++asks;
                        asked = false;
                        more = launch_control_answer(smem_u32(answer), x, y);
                        fence_proxy_async_smem();   // the answer is read before the next one may be written
                        // kEither: a CTA past the units of two heads had nothing to run, and there may be more
                        if (!(kEither && more && !single && y >= prm.num_q_tiles)) break;
                        ask();
                    }
                    if (!ok) break;
                }
            }
            // copies still in flight must land before the CTA's shared memory is released (CG 2: the first
            // CTA sees both CTAs' land, and both stay until the cluster barrier below; after a wait that
            // ran out the other CTA may never issue its part, so the copies get a millisecond to land)
            if (asked) mbar_wait_bounded(bar(C::B_NEXT), asks & 1, prm.err, 27);
            if (CG == 2 && *abort_flag) {
                const uint64_t t0 = padoc_globaltimer();
                while (padoc_globaltimer() - t0 < 1000000ull) {
                }
            } else if (rank == 0) {
                for (int i = 0; i < NH; ++i)
                    if (nq[i]) mbar_wait_bounded(bar(C::B_QFULL + i), (nq[i] - 1) & 1, prm.err, 27);
                for (int t = max(tk - kStages, 0); t < tk; ++t)
                    mbar_wait_bounded(bar(C::B_KFULL + t % kStages), (t / kStages) & 1, prm.err, 28);
                for (int t = max(tv - kStages, 0); t < tv; ++t)
                    mbar_wait_bounded(bar(C::B_VFULL + t % kStages), (t / kStages) & 1, prm.err, 29);
            }
        } else if (warp >= 9 && warp < 9 + (single ? 1 : NH) && rank == 0) {
            // ------------------------------------------------------------ MMA issuers (a whole warp per head)
            const int i = warp - 9;
            constexpr uint32_t idS = umma_idesc_bf16(128 * CG, 64, false);
            constexpr uint32_t idPV = umma_idesc_bf16(128 * CG, kD, true);
            const uint64_t dq = umma_desc_sw128(smem_u32(sq + i * kTile), 16, 1024);
            const uint64_t dk = umma_desc_sw128(smem_u32(sk), 16, 1024), dv = umma_desc_sw128(smem_u32(sv), kPanel, 1024);
            const uint32_t tS = tmem + 128 * i, tO = tmem + 256 + 128 * i;
            auto wait = [&](int b, uint32_t parity, int site) {
                return mbar_wait_warp(bar(b), parity, prm.err, site, abort_flag);
            };
            auto commit = [&](int b) {
                if (CG == 2) umma_commit_pair_warp(bar(b));
                else umma_commit_warp(bar(b));
            };
            // S_i over half h of the tile in the given stage; the last tile of a unit frees Q_i
            auto issue_s = [&](int stage, int h, bool last) {
                umma_bf16_ss_k128_warp<CG, kPanel, C::kKPanel>(tS + 64 * h, dq, dk + ((stage * C::kHalf + h * 2 * C::kKPanel) >> 4),
                                                               idS);
                commit(C::B_SFULL + 2 * i + h);
                if (h == 1) {
                    if (last) commit(C::B_QEMPTY + i);
                    commit(C::B_KEMPTY + stage);
                }
            };
            int n = 0;   // units read
            // entries of the next unit that has any (0: none left), false when a wait ran out
            auto next_unit = [&](int &ne) {
                Unit u;
                do {
                    if (!read_unit(n++, u, 30)) return false;
                } while (u.ne == 0);
                ne = max(u.ne, 0);
                return true;
            };
            int ne = 0, t = 0;   // t: tiles over all units
            bool ok = next_unit(ne);
            if (ok && ne > 0) {
                ok = wait(C::B_KFULL, 0, 31) && wait(C::B_QFULL + i, 0, 32);
                if (ok) {
                    tc_fence_after();
                    issue_s(0, 0, ne == 1);
                    issue_s(0, 1, ne == 1);
                }
            }
            // O_i += P_i V over half h of tile t
            auto issue_pv = [&](int s, int h, bool first) {
                if (!wait(C::B_PFULL + 2 * i + h, t & 1, 35)) return false;
                tc_fence_after();
                umma_bf16_ts_k64_mn_warp<CG>(tO, tS + 64 * h, dv + ((s * C::kHalf + h * 8192) >> 4), idPV, !first);
                commit(C::B_PVDONE + 2 * i + h);
                if (h == 1) commit(C::B_VEMPTY + s);
                return true;
            };
            for (int w = 0; ok && ne > 0; ++w) {
                if (w > 0) ok = wait(C::B_OFREE + i, (w - 1) & 1, 34);
                for (int j = 0; ok && j + 1 < ne; ++j, ++t) {
                    const int s = t % kStages, sn = (t + 1) % kStages;
                    // (while the tensor cores still run the S of this tile)
                    ok = wait(C::B_VFULL + s, (t / kStages) & 1, 33) && wait(C::B_KFULL + sn, ((t + 1) / kStages) & 1, 36);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (ok && (ok = issue_pv(s, h, j == 0 && h == 0))) issue_s(sn, h, j + 2 == ne);
                }
                if (!ok) break;
                // the unit's last tile, then the first S of the next unit, under this one's epilogue
                const int s = t % kStages;
                ok = wait(C::B_VFULL + s, (t / kStages) & 1, 33) && issue_pv(s, 0, ne == 1) && issue_pv(s, 1, false);
                if (!ok) break;
                ++t;
                ok = next_unit(ne);
                if (!ok || ne == 0) break;
                ok = wait(C::B_KFULL + t % kStages, (t / kStages) & 1, 36) && wait(C::B_QFULL + i, (w + 1) & 1, 37);
                if (ok) {
                    tc_fence_after();
                    issue_s(t % kStages, 0, ne == 1);
                    issue_s(t % kStages, 1, ne == 1);
                }
            }
            // every MMA issued above must complete before TMEM is released
            if (CG == 2) umma_commit_pair_warp(bar(C::B_FINAL + i));
            else umma_commit_warp(bar(C::B_FINAL + i));
            mbar_wait_bounded(bar(C::B_FINAL + i), 0, prm.err, 38);
        }
    } else if (warp / 4 < (single ? 1 : NH)) {
        // ---------------------------------------------------------------- softmax + epilogue
        const int hi = warp / 4;                    // head index inside the unit
        const int row = tid & 127;
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lanes + 128 * hi, tO = tmem + lanes + 256 + 128 * hi;
        const float c = prm.scale_log2;
        // every decision below is warp-uniform: the TMEM loads and stores are warp-collective
        auto wait_all = [&](int b, uint32_t parity, int site) {
            return mbar_wait_warp(bar(b), parity, prm.err, site, abort_flag);
        };
        bool ok = true;
        int t_tile = 0;   // tiles so far
        // the next unit with entries and what its first tile needs, read before the previous one's output
        // is written; ne 0: none left
        Unit u;
        int n = 0, kt_next = 0, kind_next = 0;
        int4 span = make_int4(0, 0, 0, 0);
        auto next_unit = [&]() {
            do {
                if (!read_unit(n++, u, 39)) return false;
            } while (u.ne == 0);
            u.ne = max(u.ne, 0);
            if (u.ne == 0) return true;
            const int64_t t = (int64_t)u.qt * kQT + row;
            span = t < prm.T ? *reinterpret_cast<const int4 *>(prm.spans + 4 * t) : make_int4(0, 0, 0, 0);
            kt_next = prm.tile_k[u.e0];
            kind_next = prm.tile_kind[u.e0];
            return true;
        };
        ok = next_unit();
        while (ok && u.ne > 0) {
            const int ne = u.ne, e0 = u.e0, h = u.h0 + NH * (int)rank + hi, qrow = u.qt * kQT + (warp & 3) * 32;
            const int a0 = span.x, a1 = span.y, b0 = span.z, b1 = span.w;
            float m_ref = -INFINITY, l = 0.f;   // m_ref in raw score units
            for (int j = 0; j < ne; ++j, ++t_tile) {
                const int kt = kt_next;
                const bool full = kind_next == PADOC_TILE_FULL;   // the same for every row of the CTA
                if (j + 1 < ne) { kt_next = prm.tile_k[e0 + j + 1]; kind_next = prm.tile_kind[e0 + j + 1]; }
                const int cb = kt * kKT;
                const int lo0 = clamp_tile(a0 - cb), w0 = max(clamp_tile(a1 - cb) - lo0, 0);
                const int lo1 = clamp_tile(b0 - cb), w1 = max(clamp_tile(b1 - cb) - lo1, 0);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint32_t tB = tS + 64 * half;
                    if (!wait_all(C::B_SFULL + 2 * hi + half, t_tile & 1, 40)) { ok = false; break; }
                    tc_fence_after();
                    // the row's scores are read from tensor memory once and stay in registers
                    uint32_t sr[2][32];
                    tmem_ld32(tB, sr[0]);
                    tmem_ld32(tB + 32, sr[1]);
                    tmem_ld_wait();
                    float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if (!full) {
                            const int base = 64 * half + 32 * q;
                            const uint32_t vis = interval_bits(lo0, w0, base) | interval_bits(lo1, w1, base);
                            if (__any_sync(0xffffffffu, vis != 0xffffffffu)) {
#pragma unroll
                                for (int i = 0; i < 32; ++i) sr[q][i] = (vis >> i) & 1u ? sr[q][i] : 0xff800000u;   // -inf
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 32; i += 8) {
                            mx4[0] = fmax3f(mx4[0], __uint_as_float(sr[q][i]), __uint_as_float(sr[q][i + 1]));
                            mx4[1] = fmax3f(mx4[1], __uint_as_float(sr[q][i + 2]), __uint_as_float(sr[q][i + 3]));
                            mx4[2] = fmax3f(mx4[2], __uint_as_float(sr[q][i + 4]), __uint_as_float(sr[q][i + 5]));
                            mx4[3] = fmax3f(mx4[3], __uint_as_float(sr[q][i + 6]), __uint_as_float(sr[q][i + 7]));
                        }
                    }
                    const float mx = fmaxf(fmax3f(mx4[0], mx4[1], mx4[2]), mx4[3]);
                    const float m_new = fmaxf(m_ref, mx);
                    // a row with nothing accumulated yet (O holds zeros) adopts the new maximum directly;
                    // otherwise the reference only moves when the maximum grew by more than 2^8
                    const bool rescale = m_ref != -INFINITY && (m_new - m_ref) * c > 8.f;
                    if (m_ref == -INFINITY) m_ref = m_new;
                    if (__any_sync(0xffffffffu, rescale)) {
                        // O_i is quiescent once the previous half's PV is done: the next one waits for this P
                        // (the one before that was done before this half's S)
                        if (!wait_all(C::B_PVDONE + 2 * hi + (half ^ 1), (half ? t_tile : t_tile - 1) & 1, 41)) { ok = false; break; }
                        tc_fence_after();
                        const float alpha = rescale ? fast_exp2((m_ref - m_new) * c) : 1.f;
#pragma unroll 1   // (rare; unrolled it takes registers from every tile)
                        for (int q = 0; q < 8; ++q) {
                            uint32_t o[16];
                            tmem_ld16(tO + q * 16, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tmem_st16(tO + q * 16, o);
                        }
                        if (rescale) { l *= alpha; m_ref = m_new; }
                    }
                    const float moff = m_ref == -INFINITY ? 0.f : m_ref * c;
                    // P = exp2(S * c - m * c) as packed bf16 over the first 32 columns of this half's S
                    const uint64_t c2 = f2_pack(c, c), moff2 = f2_pack(-moff, -moff);
                    uint64_t rs[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint32_t pk[16];
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            float x0, x1;
                            f2_unpack(f2_fma(f2_pack(__uint_as_float(sr[q][i]), __uint_as_float(sr[q][i + 1])), c2, moff2), x0, x1);
                            const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                            rs[(i >> 1) & 3] = f2_add(rs[(i >> 1) & 3], f2_pack(p0, p1));
                            pk[i >> 1] = pack_bf16x2(p0, p1);
                        }
                        tmem_st16(tB + q * 16, pk);
                    }
                    float r0, r1;
                    f2_unpack(f2_add(f2_add(rs[0], rs[1]), f2_add(rs[2], rs[3])), r0, r1);
                    l += r0 + r1;
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_lead(C::B_PFULL + 2 * hi + half);
                }
                if (!ok) break;
            }
            const int last_tile = t_tile - 1;
            if (!ok || !(ok = next_unit()) || !(ok = wait_all(C::B_PVDONE + 2 * hi + 1, last_tile & 1, 43))) break;
            tc_fence_after();
            // O / l through shared memory and the TMA, 64 dims of the warp's 32 rows at a time (rows past T
            // are not written); O_i is free for the next unit's PV as soon as it is read
            const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint8_t *stage = so + (warp * C::kOutPanels + half % C::kOutPanels) * 4096;
                if (half < C::kOutPanels ? half == 0 : true) {   // the staging's last copies have read it
                    if (lane == 0) tma_store_wait_read<0>();
                    __syncwarp();
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    uint32_t o[32];
                    tmem_ld32(tO + 64 * half + 32 * q, o);
                    tmem_ld_wait();
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint4 x;
                        x.x = pack_bf16x2(__uint_as_float(o[8 * k]) * inv, __uint_as_float(o[8 * k + 1]) * inv);
                        x.y = pack_bf16x2(__uint_as_float(o[8 * k + 2]) * inv, __uint_as_float(o[8 * k + 3]) * inv);
                        x.z = pack_bf16x2(__uint_as_float(o[8 * k + 4]) * inv, __uint_as_float(o[8 * k + 5]) * inv);
                        x.w = pack_bf16x2(__uint_as_float(o[8 * k + 6]) * inv, __uint_as_float(o[8 * k + 7]) * inv);
                        *reinterpret_cast<uint4 *>(stage + lane * 128 + (((4 * q + k) ^ (lane & 7)) << 4)) = x;
                    }
                }
                if (half == 1) tc_fence_before();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (half == 1) arrive_lead(C::B_OFREE + hi);
                    tma_store_2d(&omap, h * kD + 64 * half, qrow, smem_u32(stage));
                    tma_store_commit();
                }
            }
            if (qrow + lane < prm.T)
                prm.lse[(size_t)(qrow + lane) * prm.num_q_heads + h] = l > 0.f ? (m_ref * c + log2f(l)) * PADOC_LN2 : -INFINITY;
        }
        if (lane == 0) tma_store_wait_read<0>();   // before the CTA's shared memory is released
    }
    tc_fence_before();
    __syncthreads();
    // neither CTA leaves while the other may still reach its shared memory, barriers or tensor memory
    if (CG == 2) cluster_sync();
    if (warp == 9) {
        tc_fence_after();
        tmem_dealloc<CG>(tmem, kTmemCols);
    }
}

template <int NH, int CG, bool kEither = false>
padoc_status launch(const CUtensorMap &qmap, const CUtensorMap &kmap, const CUtensorMap &vmap, const CUtensorMap &omap,
                    const TcPrefillParams &prm,
                    unsigned nqt, cudaStream_t stream)
{
    auto kernel = prefill_tc_kernel<NH, CG, kEither>;
    constexpr size_t bytes = Cfg<NH, CG>::kSmemBytes;
    if (const padoc_status st = padoc_set_max_smem((const void *)kernel, (int)bytes)) return st;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(prm.num_q_heads / NH), kEither ? 2 * nqt : nqt);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = bytes;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CG;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = CG == 1 ? 0 : 1;   // (304 single CTAs as clusters of one took 15.9 us, as plain ones 14.1)
    PADOC_CUDA_TRY(cudaLaunchKernelEx(&lc, kernel, qmap, kmap, vmap, omap, prm));
    return padoc_launch_status();
}


}  // namespace

padoc_status padoc_launch_prefill_tc(const void *q, const void *k, const void *v, int64_t total_tokens,
                                     int32_t num_q_heads, int32_t num_kv_heads, const int32_t *spans_dev,
                                     const int32_t *tile_row_ptr_dev, const int32_t *tile_k_dev,
                                     const int8_t *tile_kind_dev, float scale_log2, void *out, float *lse,
                                     cudaStream_t stream)
{
    int *err = padoc_device_error_word();
    if (!err) return PADOC_ERR_CUDA;
    const int64_t nqt = (total_tokens + kQT - 1) / kQT;
    if (nqt > 65535) return PADOC_ERR_UNSUPPORTED;
    // Up to one (q-tile, head) unit an SM, a CTA per unit: the call lasts as long as its longest unit, and a head
    // alone takes ~1000 cycles a half where two share the tensor cores (1450). Up to two an SM that is right
    // while the longest units set the time, but short units then come in two waves where two heads a CTA need
    // one: the kernel decides by the map (one_head_units, fitted to 175 calls timed with both: within 0.4% of the
    // better one on the mean, 12% at most). At 256 units, 16 / 2 heads, one head / two heads a CTA: 2045 tokens
    // as one causal page 24.2 / 30.8 us, as 12 short pages 15.7 / 11.9. Above two an SM, CTA pairs when the heads
    // of a KV head come in fours (34107 tokens: 332 us against 400 with two heads on a CTA), else two or one.
    const int group = num_q_heads / num_kv_heads;
    const int64_t units = nqt * num_q_heads, sms = padoc_default_ctas();
    const bool small = units <= (group % 2 == 0 ? sms : 2 * sms), either = !small && units <= 2 * sms && nqt <= kEitherTiles;
    const int cg = !small && !either && group % 4 == 0 ? 2 : 1;
    CUtensorMap qmap, kmap, vmap, omap;
    if (!padoc_make_tmap_bf16(&qmap, q, (uint64_t)num_q_heads * kD, total_tokens, (uint64_t)num_q_heads * kD * 2, 64, kQT) ||
        !padoc_make_tmap_bf16(&kmap, k, (uint64_t)num_kv_heads * kD, total_tokens, (uint64_t)num_kv_heads * kD * 2, 64, 64 / cg) ||
        !padoc_make_tmap_bf16(&vmap, v, (uint64_t)num_kv_heads * kD, total_tokens, (uint64_t)num_kv_heads * kD * 2, 64, kKT) ||
        !padoc_make_tmap_bf16(&omap, out, (uint64_t)num_q_heads * kD, total_tokens, (uint64_t)num_q_heads * kD * 2, 64, 32))
        return PADOC_ERR_CUDA;
    TcPrefillParams prm;
    prm.spans = spans_dev;
    prm.row_ptr = tile_row_ptr_dev;
    prm.tile_k = tile_k_dev;
    prm.tile_kind = tile_kind_dev;
    prm.T = total_tokens;
    prm.num_q_heads = num_q_heads;
    prm.num_kv_heads = num_kv_heads;
    prm.num_q_tiles = (int32_t)nqt;
    prm.over = (float)units / (float)sms - 1.f;
    prm.scale_log2 = scale_log2;
    prm.lse = lse;
    prm.err = err;
    if (either) return launch<2, 1, true>(qmap, kmap, vmap, omap, prm, (unsigned)nqt, stream);
    if (cg == 2) return launch<2, 2>(qmap, kmap, vmap, omap, prm, (unsigned)nqt, stream);
    if (!small && group % 2 == 0) return launch<2, 1>(qmap, kmap, vmap, omap, prm, (unsigned)nqt, stream);
    return launch<1, 1>(qmap, kmap, vmap, omap, prm, (unsigned)nqt, stream);
}
