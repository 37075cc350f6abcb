// e4m3.cu -- writing the FP8 (E4M3) variant of the paged KV cache (C5): whole blocks quantized at
// once (a page's prefix after its prefill), and one row per input appended by a decoding loop
// (Algorithm 1's "Append i to the cache", App. E.1). The paper serves a bf16 cache; this variant
// stores K and V as E4M3 codes with one fp32 scale per (block, KV head), the scale being amax / 448
// over the rows the block holds, so that a block's largest magnitude maps to the format's largest
// finite value. All arithmetic that decides a code is fp32 with round-to-nearest-even (division and
// product rounded once each), so the codes are a function of the inputs alone.
#include "common.cuh"
#include "tc.cuh"

namespace {

constexpr int kD = 128;        // head_dim of the E4M3 path
constexpr int kBlk = 16;       // tokens per block
constexpr int kQuantWarps = 8;  // warps per CTA of the quantize kernel, one (block, head, K or V) each

// x / s rounded to fp32, for many x and one s. Both kernels are bound by arithmetic, not memory, when
// every value pays an IEEE division of its own. With inv = 1 / s correctly rounded and q within one unit
// of the last place of x / s, r = x - q s is exact and q + r inv, rounded once, is x / s correctly rounded
// (Markstein 1990, theorem on the final division step); the first such step brings x inv within that unit,
// the second rounds: five packed instructions for two values. Exact for 2^-80 < s < 2^80 and every
// |x / s| >= 2^-20 (smaller quotients have the code 0 with or without the last rounding): q is a multiple
// of 2^-43 and s of 2^-103, so r is one of 2^-146 and is held exactly, as a subnormal too: the packed
// instructions must not flush them. Other scales take the division.
struct Scale {
    float s, inv;
    bool fast;
    // the codes of two values (x0 in the low byte)
    __device__ __forceinline__ uint32_t codes(float x0, float x1) const
    {
        float y0, y1;
        if (fast) {
            const uint64_t x = f2_pack(x0, x1), i2 = f2_pack(inv, inv), n2 = f2_pack(-s, -s);
            uint64_t q = f2_mul(x, i2);
            q = f2_fma(f2_fma(q, n2, x), i2, q);
            f2_unpack(f2_fma(f2_fma(q, n2, x), i2, q), y0, y1);
            y0 = copysignf(y0, x0);   // (-0, which the steps turn into +0, keeps its code)
            y1 = copysignf(y1, x1);
        } else {
            y0 = __fdiv_rn(x0, s);
            y1 = __fdiv_rn(x1, s);
        }
        return f32x2_to_e4m3x2(y0, y1);
    }
};

__device__ __forceinline__ Scale make_scale(float s)
{
    return Scale{s, __frcp_rn(s), s > 0x1p-80f && s < 0x1p80f};
}

__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, sh));
    return v;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// One warp per (source block i, head g, K or V): k_src or v_src ([count][Hkv][16][128] bf16) becomes
// (block dst_blocks[i], head g) of the pool: scale = amax / 448, codes of x / scale (0 and codes 0 for
// an all-zero one). A lane holds eight 16-byte pieces, one of each 512 bytes, so that the warp's loads
// (all in flight at once) and its code stores cover whole lines, and the maximum needs shuffles only.
// Bound by HBM (70% of its rate) once the arithmetic is cheap: 12168 blocks x 2 heads (300 MB) took
// 67 us with a CTA of 128 threads, two barriers and a division a value per block; now 44 us.
__global__ void __launch_bounds__(32 * kQuantWarps) quantize_blocks_kernel(
    const uint4 *__restrict__ k_src, const uint4 *__restrict__ v_src, const int32_t *__restrict__ dst_blocks,
    uint8_t *__restrict__ k_codes, uint8_t *__restrict__ v_codes, float *__restrict__ k_scales, float *__restrict__ v_scales,
    int64_t units, int32_t num_blocks, int32_t hkv, int *err)
{
    // a programmatic dependent of the previous kernel in the stream, as the append
    pdl_wait_prerequisite();
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31;
    int64_t u = (int64_t)blockIdx.x * kQuantWarps + (threadIdx.x >> 5);
    if (u >= 2 * units) return;
    const bool is_v = u >= units;
    if (is_v) u -= units;
    const uint4 *src = (is_v ? v_src : k_src) + u * (kBlk * kD / 8) + lane;
    uint4 w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = __ldcs(src + 32 * k);
    const int64_t i = u / hkv;
    const int g = (int)(u - i * hkv);
    const int32_t b = dst_blocks[i];
    if (b < 0 || b >= num_blocks) {
        if (lane == 0 && g == 0 && !is_v) padoc_record_error(err, PADOC_DEVERR_BLOCK_ID, b);
        return;
    }
    __nv_bfloat162 m = __float2bfloat162_rn(0.f);   // (the maximum of bf16 magnitudes is one of them: exact)
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t x[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) m = __hmax2(m, __habs2(*reinterpret_cast<const __nv_bfloat162 *>(&x[j])));
    }
    const float a = fmaxf(__low2float(m), __high2float(m));
    const Scale sc = make_scale(__fdiv_rn(warp_max(a), 448.f));
    if (lane == 0) (is_v ? v_scales : k_scales)[(size_t)b * hkv + g] = sc.s;
    uint2 *dst = reinterpret_cast<uint2 *>((is_v ? v_codes : k_codes) + ((size_t)b * hkv + g) * kBlk * kD) + lane;
    if (!(sc.s > 0.f)) {
#pragma unroll
        for (int k = 0; k < 8; ++k) dst[32 * k] = make_uint2(0u, 0u);
        return;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t x[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
        uint32_t c[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = sc.codes(bf16_lo(x[j]), bf16_hi(x[j]));
        dst[32 * k] = make_uint2(c[0] | c[1] << 16, c[2] | c[3] << 16);
    }
}

// One CTA of 4 warps per input i: its K and V rows (row src_rows[i] of k_src / v_src, [src_total][Hkv][128]
// bf16) go to row r = slots[i] % 16 of block slots[i] / 16, every KV head, by the scale rule: the
// new scale is max(old, amax(row) / 448) (the old one taken as 0 at r = 0, which starts a block
// afresh); when it grows from a nonzero old scale, rows 0 .. r-1 are re-encoded (code value x old
// scale, then / new scale, each rounded to fp32); the row's codes are those of x / new scale. The
// query row goes to row i of q_dst. A warp takes a (K or V, head) at a time and a lane four dims, with
// the block's earlier rows loaded before the maximum is known: latency-bound, one load latency instead
// of one per row (630 inputs: 20 us when a CTA took the heads in turn and re-read a row per step, 7 us now).
constexpr int kAppendWarps = 4;
template <bool kAligned>
__device__ __forceinline__ uint32_t load_codes(const uint8_t *p)
{
    if (kAligned) return *reinterpret_cast<const uint32_t *>(p);
    return p[0] | p[1] << 8 | p[2] << 16 | (uint32_t)p[3] << 24;
}
template <bool kAligned>
__device__ __forceinline__ void store_codes(uint8_t *p, uint32_t c)
{
    if (kAligned) *reinterpret_cast<uint32_t *>(p) = c;
    else
        for (int j = 0; j < 4; ++j) p[j] = (uint8_t)(c >> (8 * j));
}

// kAligned: the pool's codes start on 4-byte boundaries (the append also takes pools that do not)
template <bool kAligned>
__global__ void __launch_bounds__(32 * kAppendWarps) append_e4m3_kernel(
    const __nv_bfloat16 *__restrict__ k_src, const __nv_bfloat16 *__restrict__ v_src, const uint4 *__restrict__ q_src,
    int64_t src_total, uint4 *__restrict__ q_dst, const int32_t *__restrict__ src_rows, const int32_t *__restrict__ slots,
    uint8_t *k_codes, uint8_t *v_codes, float *k_scales, float *v_scales, int64_t pool_slots, int32_t hkv, int32_t hq, int *err)
{
    // a programmatic dependent of the previous kernel in the stream, as the bf16 append
    pdl_wait_prerequisite();
    pdl_launch_dependents();
    const int64_t i = blockIdx.x;
    const int64_t row = src_rows ? (int64_t)src_rows[i] : i;
    const int64_t slot = slots[i];
    if (slot < 0 || slot >= pool_slots || row < 0 || row >= src_total) {
        if (threadIdx.x == 0)
            padoc_record_error(err, PADOC_DEVERR_BLOCK_ID, (slot < 0 || slot >= pool_slots) ? (int)slot : (int)row);
        return;
    }
    const int64_t blk = slot / kBlk;
    const int r = (int)(slot % kBlk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int u = warp; u < 2 * hkv; u += kAppendWarps) {
        const bool is_v = u >= hkv;
        const int g = is_v ? u - hkv : u;
        float *scp = (is_v ? v_scales : k_scales) + blk * hkv + g;
        uint8_t *codes = (is_v ? v_codes : k_codes) + (blk * hkv + g) * kBlk * kD + 4 * lane;
        const uint2 w = *(reinterpret_cast<const uint2 *>((is_v ? v_src : k_src) + (row * hkv + g) * kD) + lane);
        const float s_old = r == 0 ? 0.f : *scp;
        uint32_t old[kBlk - 1];
#pragma unroll
        for (int rr = 0; rr < kBlk - 1; ++rr) old[rr] = rr < r ? load_codes<kAligned>(codes + rr * kD) : 0u;
        const float x[4] = {bf16_lo(w.x), bf16_hi(w.x), bf16_lo(w.y), bf16_hi(w.y)};
        const float a = warp_max(fmaxf(fmaxf(fabsf(x[0]), fabsf(x[1])), fmaxf(fabsf(x[2]), fabsf(x[3]))));
        const float cand = __fdiv_rn(a, 448.f);
        const Scale sc = make_scale(cand > s_old ? cand : s_old);
        if (sc.s > s_old && s_old > 0.f) {
#pragma unroll
            for (int rr = 0; rr < kBlk - 1; ++rr) {
                if (rr >= r) break;
                float y[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) y[j] = __fmul_rn(e4m3_to_f32((uint8_t)(old[rr] >> (8 * j))), s_old);
                store_codes<kAligned>(codes + rr * kD, sc.codes(y[0], y[1]) | sc.codes(y[2], y[3]) << 16);
            }
        }
        store_codes<kAligned>(codes + r * kD, sc.s > 0.f ? sc.codes(x[0], x[1]) | sc.codes(x[2], x[3]) << 16 : 0u);
        __syncwarp();   // every lane has read the old scale before it is replaced
        if (lane == 0) *scp = sc.s;
    }
    if (q_src) {
        const int q_vecs = hq * (kD * 2 / 16);
        const uint4 *qs = q_src + row * q_vecs;
        uint4 *qd = q_dst + i * q_vecs;
        for (int c = threadIdx.x; c < q_vecs; c += 32 * kAppendWarps) qd[c] = qs[c];
    }
}

bool e4m3_pool_ok(const padoc_kv_pool_e4m3 *pool)
{
    return pool && pool->k_codes && pool->v_codes && pool->k_scales && pool->v_scales && pool->num_blocks >= 1 &&
           pool->num_kv_heads >= 1 && pool->block_size >= 1 && pool->head_dim >= 1;
}

}  // namespace

extern "C" padoc_status padoc_quantize_kv_blocks(const padoc_kv_pool_e4m3 *pool, const void *k_src, const void *v_src,
                                                 const int32_t *dst_blocks, int32_t count, padoc_stream_t stream)
{
    if (!e4m3_pool_ok(pool) || count < 0) return PADOC_ERR_INVALID_ARGUMENT;
    if (pool->block_size != kBlk || pool->head_dim != kD || pool->num_kv_heads > 65535) return PADOC_ERR_UNSUPPORTED;
    if (count == 0) return PADOC_OK;
    if (!k_src || !v_src || !dst_blocks) return PADOC_ERR_INVALID_ARGUMENT;
    const uintptr_t align = (uintptr_t)pool->k_codes | (uintptr_t)pool->v_codes | (uintptr_t)k_src | (uintptr_t)v_src;
    if ((align & 15) || (((uintptr_t)pool->k_scales | (uintptr_t)pool->v_scales) & 3)) return PADOC_ERR_INVALID_ARGUMENT;
    int *err = padoc_device_error_word();
    if (!err) return PADOC_ERR_CUDA;
    const int64_t units = (int64_t)count * pool->num_kv_heads;   // of K, and as many of V
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)((2 * units + kQuantWarps - 1) / kQuantWarps));
    lc.blockDim = dim3(32 * kQuantWarps);
    lc.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see the kernel's wait
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    PADOC_CUDA_TRY(cudaLaunchKernelEx(&lc, quantize_blocks_kernel, (const uint4 *)k_src, (const uint4 *)v_src, dst_blocks,
                                      (uint8_t *)pool->k_codes, (uint8_t *)pool->v_codes, (float *)pool->k_scales,
                                      (float *)pool->v_scales, units, pool->num_blocks, pool->num_kv_heads, err));
    return padoc_launch_status();
}

extern "C" padoc_status padoc_append_inputs_e4m3(const padoc_kv_pool_e4m3 *pool, const void *k_src, const void *v_src,
                                                 const void *q_src, int64_t src_total, int32_t num_q_heads, void *q_dst,
                                                 const int32_t *src_rows, const int32_t *slots, int32_t count,
                                                 padoc_stream_t stream)
{
    if (!e4m3_pool_ok(pool) || count < 0 || src_total < 0) return PADOC_ERR_INVALID_ARGUMENT;
    if (pool->block_size != kBlk || pool->head_dim != kD) return PADOC_ERR_UNSUPPORTED;
    if (count == 0) return PADOC_OK;
    if (!k_src || !v_src || !slots) return PADOC_ERR_INVALID_ARGUMENT;
    if (q_src && (!q_dst || num_q_heads < 1)) return PADOC_ERR_INVALID_ARGUMENT;
    const uintptr_t align = (uintptr_t)k_src | (uintptr_t)v_src | (uintptr_t)q_src | (uintptr_t)q_dst;
    if ((align & 15) || (((uintptr_t)pool->k_scales | (uintptr_t)pool->v_scales) & 3)) return PADOC_ERR_INVALID_ARGUMENT;
    int *err = padoc_device_error_word();
    if (!err) return PADOC_ERR_CUDA;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)count);
    lc.blockDim = dim3(32 * kAppendWarps);
    lc.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see the kernel's wait
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    const bool aligned = !(((uintptr_t)pool->k_codes | (uintptr_t)pool->v_codes) & 3);
    PADOC_CUDA_TRY(cudaLaunchKernelEx(&lc, aligned ? append_e4m3_kernel<true> : append_e4m3_kernel<false>, (const __nv_bfloat16 *)k_src, (const __nv_bfloat16 *)v_src,
                                      (const uint4 *)q_src, src_total, (uint4 *)q_dst, src_rows, slots,
                                      (uint8_t *)pool->k_codes, (uint8_t *)pool->v_codes, (float *)pool->k_scales,
                                      (float *)pool->v_scales, (int64_t)pool->num_blocks * kBlk, pool->num_kv_heads,
                                      q_src ? num_q_heads : 0, err));
    return padoc_launch_status();
}
