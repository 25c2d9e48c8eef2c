// LSH-DIN without a pass over the pairs (sm_100a; Section 4.2, eqs. 6-8): for requests of many keys and candidates.
//
// eq. 8 weighs every sequence row by a match count, and match counts are linear in the candidate's signature: with bits as q_i,
// s_ki = +-1, 2 matches_k = d' + sum_i q_i s_ki, so
//     sum_k (2 matches_k) S_k = d' sum_k S_k + sum_i q_i A_i,   A_i = sum_k s_ki S_k.
// A and the sum of the rows depend on the request alone: [d' + 1 x d] numbers.  What a candidate costs then does not grow with the
// sequence: [1 x d'] . [d' x d] instead of [1 x L] . [L x d] and the conversion of L match counts into an operand.  16 requests of 10^4
// candidates and 10^4 keys, d 128: 15 + 12 us, and 215 for SimTier's counts alone (aif_tc_tier.cu), in place of 650 for the pass over the pairs that
// yields both.
//
//   k_din_sums    A and the row sums per request, on the tensor cores: a cluster of up to eight CTAs shares a request's key blocks,
//                 leaves its partial sums in global memory, and after a cluster barrier every CTA adds an eighth of the numbers in
//                 the order of the pieces and writes them as the next kernel's operand: every number split into three bf16 parts
//                 (24 bits: nothing of the fp32 sum is lost), K-major, in the swizzled layout of shared memory.
//   k_din_apply   rows = [q, q, q, 1 1 1] . [A parts; d' sum parts], q exact in bf16, fp32 accumulation; scaled and stored.
//
// A sequence row that is not finite makes the row sums of its columns infinite or NaN, and the A of its columns infinite with either sign.  A NaN
// sum is the column's value for every candidate.  Where the sum is an infinity, every match count but zero hands that on, and zero times it is
// NaN: A_i's sign is the row's bit, so the operand takes signs (0 where several such rows differ in a bit) and d' in place of the sum, the
// product is twice the row's match count (positive if rows with different bits are behind it), and the rows' columns are multiplied by the
// infinity when they leave.  (Several infinite rows of different bits, one of them the complement of the candidate's: the infinity.)
#include <type_traits>

#include "aif_device.cuh"
#include "aif_internal.h"
#include "aif_tc_ptx.cuh"

namespace aif {
namespace {

constexpr int kDinBlock = 128;    // keys per block
constexpr int kDinCols = 128;     // columns of S per CTA (k_din_sums) or item (k_din_apply)
constexpr int kDinCluster = 8;    // most CTAs that share a request's keys
constexpr int kDinRequests = 256; // requests at a time (29 MB of operands at d = 128, 109 at 256): a launch of more goes in rounds of as many

__host__ __device__ constexpr int din_chunks(int D) { return 3 * (D / 64) + 1; }                     // 64-wide K chunks of the operand
__host__ __device__ constexpr size_t din_image_bytes(int D) { return (size_t)din_chunks(D) * D * 128; }   // of a request
__host__ __device__ constexpr size_t din_image_step(int D) { return din_image_bytes(D) + 128; }   // behind it: per 32 columns, which are infinite, and negative
__host__ __device__ constexpr int din_record_groups(int D) { return D / 4 + 1; }                     // float4 groups of a partial record, the last one the row sum
__host__ __device__ constexpr size_t din_record_bytes(int D) { return (size_t)din_record_groups(D) * kDinCols * 16; }

// As umma_idesc_bf16_bmn, with A MN-major too (bit 15).
__host__ __device__ constexpr uint32_t umma_idesc_bf16_mn_mn(int m, int n) { return umma_idesc_bf16_bmn(m, n) | (1u << 15); }

struct DinSums {
    const SlotDev *slots;
    const ReqDev *reqs;     // the requests at hand, or nullptr: single
    ReqDev single;
    int32_t parts;          // CTAs per request and column half = cluster size
    int32_t late;
    uint32_t *status;
    float4 *records;        // [request][column half][part] records
    unsigned char *image;   // [request] operands
};

template <int D>
struct DinSumsCfg {
    static constexpr int kStages = D <= 128 ? 3 : 2;
    // Shared memory in chunks of 16 KB (128 keys x 128 bytes).  The operands' 64-element groups may lie any fixed distance apart, so at d = 128
    // every stage's two signature groups and the one chunk of ones are equidistant: the row sums are sixteen more columns of the
    // same product (as products of their own, N = 16, they took 1250 cycles per block with the others, so 700).  d = 256: 256 columns are
    // the most a product has.
    static constexpr bool kOneProduct = D <= 128;
    static constexpr int kOne = 12;                                  // chunk of ones
    __host__ __device__ static constexpr int sig_first(int s) { return kOneProduct ? (s == 0 ? 10 : s == 1 ? 6 : 4) : 4 * s; }
    __host__ __device__ static constexpr int sig_step(int s) { return kOneProduct ? (s == 0 ? 1 : s == 1 ? 3 : 4) : 1; }
    __host__ __device__ static constexpr int row_first(int s) { return kOneProduct ? (s == 0 ? 0 : s == 1 ? 2 : 5) : 8 + 2 * s; }
    __host__ __device__ static constexpr int row_step(int s) { return kOneProduct && s == 2 ? 2 : 1; }
    static constexpr int kSBytes = 2 * 16384;                        // a key block's rows, 128 columns
    static constexpr int kExpandWarps = 16, kMmaWarp = 16;   // then the TMA warp
    static constexpr int kThreads = 18 * 32;
    static constexpr int kTmemCols = D + 16 <= 256 ? 256 : 512;
    static constexpr size_t kSmem = 1024 + 13 * 16384 + 256;
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ uint4 bf16_parts8(const float (&v)[8], int part)
{
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t pair = 0u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float x = v[2 * i + h];
            __nv_bfloat16 b = __float2bfloat16_rn(x);
            for (int q = 0; q < part; ++q) {   // what the parts before leave of it (an infinite part leaves nothing)
                x = isfinite(__bfloat162float(b)) ? x - __bfloat162float(b) : 0.f;
                b = __float2bfloat16_rn(x);
            }
            pair |= (uint32_t)__bfloat16_as_ushort(b) << (16 * h);
        }
        w[i] = pair;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// 32 signature bits (first bit on top of the lowest byte) as +-1 in bf16 into 64 bytes of a 128-byte row of a swizzled tile (unit u of 16
// bytes goes to u ^ swz), units u0 .. u0 + 3; `mag`: the magnitude's pair, 0 for a row of zeros.
__device__ __forceinline__ void expand_bits32(unsigned char *row, int u0, int swz, uint32_t bits, uint32_t mag)
{
    const uint32_t sign = mag ? 0x80008000u : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint32_t x = ~bits >> (8 * u);   // bit 7 first; a set bit is +1
        uint32_t o[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) o[w] = mag | (((x << (8 + 2 * w)) & 0x8000u) | ((x << (25 + 2 * w)) & 0x80000000u)) & sign;
        *reinterpret_cast<uint4 *>(row + (((u0 + u) ^ swz) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// Grid (parts, D / 128, requests), a cluster along x.
template <int D>
__global__ void __launch_bounds__((DinSumsCfg<D>::kThreads), 1) k_din_sums(const __grid_constant__ CUtensorMap tmapS, const DinSums p)
{
    using C = DinSumsCfg<D>;
    constexpr int kS = C::kStages;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    auto chunk = [&](int i) { return base + i * 16384; };
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + 13 * 16384);
    uint64_t *s_full = bars, *g_full = bars + kS, *empty = g_full + kS, *done = empty + kS;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kS; ++s) mbar_init(smem_u32(s_full + s), 1), mbar_init(smem_u32(g_full + s), C::kExpandWarps), mbar_init(smem_u32(empty + s), 1);
        mbar_init(smem_u32(done), 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < 16384 / 16; i += C::kThreads)
        reinterpret_cast<uint4 *>(chunk(C::kOne))[i] = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
    fence_proxy_async();
    if (warp == C::kMmaWarp) tmem_alloc(smem_u32(tmem_slot), C::kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (!p.late) grid_dep_wait();
    grid_dep_launch();

    const int part = blockIdx.x, half = blockIdx.y, r = blockIdx.z;
    const int slot = p.reqs ? p.reqs[r].slot : p.single.slot;
    const SlotDev *sd = p.slots + slot;
    const int L = sd->L, nb = (L + kDinBlock - 1) / kDinBlock, parts = min(p.parts, nb);
    const int b0 = part < parts ? nb * part / parts : 0, b1 = part < parts ? nb * (part + 1) / parts : 0;
    float4 *rec0 = p.records + ((size_t)r * gridDim.y + half) * p.parts * (size_t)(din_record_groups(D) * kDinCols);

    if (b1 > b0) {
        if (warp < C::kExpandWarps) {
            // signature bits of the keys -> +-1 in bf16, MN-major: a key's 64 bits are 128 bytes.  Four threads per key; the bits of the
            // next three blocks are on their way meanwhile.
            const int key = tid >> 2, sub = tid & 3;
            constexpr int kW = D / 128, kAhead = 4;   // words of 32 bits per thread
            uint32_t bits[kAhead][kW];
            auto fetch = [&](int b, uint32_t (&v)[kW]) {
                const int row = b * kDinBlock + key;
#pragma unroll
                for (int q = 0; q < kW; ++q) v[q] = b < b1 && row < L ? __ldg(reinterpret_cast<const uint32_t *>(sd->sigS + (size_t)row * (D / 8)) + sub + 4 * q) : 0u;
            };
#pragma unroll
            for (int i = 0; i < kAhead; ++i) fetch(b0 + i, bits[i]);
            bool ok = true;
            for (int b = b0, j = 0; ok && b < b1; b += kAhead)
#pragma unroll
                for (int i = 0; i < kAhead; ++i, ++j) {
                    if (b + i >= b1) break;
                    const int s = j % kS;
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(empty + s), (uint32_t)((j / kS) & 1) ^ 1u, abort_flag)))) break;
#pragma unroll
                    for (int q = 0; q < kW; ++q) {   // (rows beyond the sequence are zero in S)
                        const int word = sub + 4 * q;
                        expand_bits32(chunk(C::sig_first(s) + (word >> 1) * C::sig_step(s)) + key * 128, (word & 1) * 4, key & 7, bits[i][q], 0x3F803F80u);
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(g_full + s));
                    fetch(b + i + kAhead, bits[i]);
                }
        } else if (warp == C::kMmaWarp) {
            if (lane == 0) {
                constexpr uint32_t idesc = umma_idesc_bf16_mn_mn(kDinCols, C::kOneProduct ? D + 16 : D), idesc_one = umma_idesc_bf16_mn_mn(kDinCols, 16);
                const uint64_t one = umma_desc_mn_sw128(smem_u32(chunk(C::kOne)), 16384);
                bool ok = true;
                for (int j = 0; ok && j < b1 - b0; ++j) {
                    const int s = j % kS;
                    ok = mbar_wait(smem_u32(s_full + s), (uint32_t)((j / kS) & 1), abort_flag) && mbar_wait(smem_u32(g_full + s), (uint32_t)((j / kS) & 1), abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t a = umma_desc_mn_sw128(smem_u32(chunk(C::row_first(s))), (uint32_t)C::row_step(s) * 16384u);
                    const uint64_t g = umma_desc_mn_sw128(smem_u32(chunk(C::sig_first(s))), (uint32_t)C::sig_step(s) * 16384u);
#pragma unroll
                    for (int kk = 0; kk < kDinBlock / 16; ++kk) {   // 16 keys further = 16 rows x 128 bytes
                        const uint64_t off = (uint64_t)(kk * (2048 >> 4));
                        umma_bf16(tmem_base, a + off, g + off, idesc, j > 0 || kk > 0 ? 1u : 0u);
                        if (!C::kOneProduct) umma_bf16(tmem_base + D, a + off, one + off, idesc_one, j > 0 || kk > 0 ? 1u : 0u);
                    }
                    umma_commit(smem_u32(empty + s));
                }
                if (ok) umma_commit(smem_u32(done));
            }
            __syncwarp();
        } else {
            if (lane == 0) {
                for (int b = b0, j = 0; b < b1; ++b, ++j) {
                    const int s = j % kS;
                    if (!mbar_wait(smem_u32(empty + s), (uint32_t)((j / kS) & 1) ^ 1u, abort_flag)) break;
                    mbar_expect_tx(smem_u32(s_full + s), (uint32_t)C::kSBytes);
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        tma_load_3d(smem_u32(chunk(C::row_first(s) + c * C::row_step(s))), &tmapS, smem_u32(s_full + s), half * kDinCols + c * 64, b * kDinBlock, slot);
                }
            }
            __syncwarp();
        }
        if (warp < 4) {
            // lane = column of S, tensor-memory column = bit; then the row sum
            if (__all_sync(0xffffffffu, mbar_wait(smem_u32(done), 0u, abort_flag))) {
                tc_fence_after();
                const uint32_t lane_base = tmem_base + ((uint32_t)(warp * 32) << 16);
                float4 *out = rec0 + (size_t)part * (din_record_groups(D) * kDinCols) + warp * 32 + lane;
                tmem_rows_out(lane_base, D, out);
                uint32_t t[32];
                tmem_ld32(lane_base + (uint32_t)D, t);
                tmem_ld_wait();
                __stcg(out + (D / 4) * kDinCols, make_float4(__uint_as_float(t[0]), 0.f, 0.f, 0.f));
                tc_fence_before();
            }
        }
    }
    __syncthreads();
    if (*abort_flag && tid == 0) atomicOr(p.status, AIF_STATUS_TIMEOUT);
    // every piece's record is written (release / acquire at cluster scope covers global memory)
    __threadfence();
    cluster_sync();
    // this CTA's share of the operand: eight bits of one column per thread and round
    const int units = D / 8 * kDinCols;
    const size_t piece = (size_t)(din_record_groups(D) * kDinCols);
    unsigned char *image = p.image + (size_t)r * din_image_step(D);
    for (int u = part * C::kThreads + tid; u < units + kDinCols; u += p.parts * C::kThreads) {
        const int c = u % kDinCols, g = u / kDinCols;   // g < D / 8: bits 8 g ..; g == D / 8: the row sum
        const float4 *src = rec0 + c;
        // all pieces' numbers are requested before the first is added
        float part_sum[kDinCluster];
        float4 a[kDinCluster], b[kDinCluster];
#pragma unroll
        for (int q = 0; q < kDinCluster; ++q) {
            const float4 *at = src + (size_t)q * piece;
            part_sum[q] = q < parts ? __ldcg(at + (size_t)(D / 4) * kDinCols).x : 0.f;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            a[q] = q < parts && g < D / 8 ? __ldcg(at + (size_t)(2 * g) * kDinCols) : zero;
            b[q] = q < parts && g < D / 8 ? __ldcg(at + (size_t)(2 * g + 1) * kDinCols) : zero;
        }
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < kDinCluster; ++q) sum += part_sum[q];
        unsigned char *row = image + (size_t)(half * kDinCols + c) * 128;
        const int swz = (half * kDinCols + c) & 7;
        if (g == D / 8) {   // (a whole warp: 32 columns)
            const uint32_t inf = __ballot_sync(0xffffffffu, isinf(sum)), neg = __ballot_sync(0xffffffffu, sum < 0.f);
            if (lane == 0) reinterpret_cast<uint2 *>(image + din_image_bytes(D))[(half * kDinCols + c) >> 5] = make_uint2(inf, neg);
            const float t[8] = {isinf(sum) ? (float)D : sum * (float)D, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            const uint32_t hi = bf16_parts8(t, 0).x & 0xFFFFu, mid = bf16_parts8(t, 1).x & 0xFFFFu, lo = bf16_parts8(t, 2).x & 0xFFFFu;
            unsigned char *dst = row + (size_t)(3 * (D / 64)) * D * 128;
            *reinterpret_cast<uint4 *>(dst + (swz << 4)) = make_uint4(hi | mid << 16, lo, 0u, 0u);
            *reinterpret_cast<uint4 *>(dst + ((1 ^ swz) << 4)) = make_uint4(0u, 0u, 0u, 0u);
            continue;
        }
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < kDinCluster; ++q)
            v[0] += a[q].x, v[1] += a[q].y, v[2] += a[q].z, v[3] += a[q].w, v[4] += b[q].x, v[5] += b[q].y, v[6] += b[q].z, v[7] += b[q].w;
        if (!isfinite(sum))
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = isinf(sum) && isinf(v[i]) ? ((v[i] > 0.f) == (sum > 0.f) ? 1.f : -1.f) : 0.f;
#pragma unroll
        for (int h = 0; h < 3; ++h)
            *reinterpret_cast<uint4 *>(row + (size_t)(h * (D / 64) + (g >> 3)) * D * 128 + (((g & 7) ^ swz) << 4)) = bf16_parts8(v, h);
    }
    if (warp == C::kMmaWarp) tmem_dealloc(tmem_base, C::kTmemCols);
    if (p.late && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) grid_dep_wait();
}

struct DinApply {
    ScoreLaunch sl;
    const uint8_t *sig;
    const unsigned char *image;
    int32_t req0, tile0, n_tiles;   // the round's first request, its tiles
    int64_t M;
    int32_t mini_batch, x_stride, x_din, din_mean;
    __nv_bfloat16 *X;
};

template <int D>
struct DinApplyCfg {
    static constexpr int kHalves = D / kDinCols;             // items per tile
    static constexpr int kABytes = D / 64 * 16384;           // signatures of a tile as bf16, K-major
    static constexpr int kABufs = 2;
    static constexpr int kChunkBytes = kDinCols * 128;
    // d = 128: a request's whole operand stays (112 KB); d = 256: chunks of it go round
    static constexpr bool kResident = D <= 128;
    static constexpr int kStages = kResident ? din_chunks(D) : 4;
    static constexpr int kOnesBytes = 128 * 32;              // the row sum's factors: 1 1 1 0 ..., K = 16
    static constexpr int kOutWarps = kResident ? 8 : 4;      // two to a quarter of the rows, or one
    static constexpr int kSlabs = 2;                         // of 2 KB per output warp
    static constexpr int kStageOut = kOutWarps * kSlabs * 2048;
    static constexpr int kMmaWarp = kOutWarps, kLoadWarp = kOutWarps + 1, kExpandWarp0 = kOutWarps + 2, kExpandWarps = 8;
    static constexpr int kThreads = (kOutWarps + 10) * 32;
    static constexpr size_t kSmem = 1024 + kABufs * kABytes + kStages * kChunkBytes + kStageOut + kOnesBytes + 256;
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

// One CTA per SM walks over a range of the tiles (a request's tiles are neighbours): at d = 128 the operand is read once per request and CTA.
// Read again for every tile, chunk by chunk, a tile took 4100 cycles for 1600 of products, most of it the issuer's seven waits and the four output warps.
template <int D>
__global__ void __launch_bounds__((DinApplyCfg<D>::kThreads), 1) k_din_apply(const __grid_constant__ CUtensorMap tmapX, const DinApply p)
{
    using C = DinApplyCfg<D>;
    constexpr int kS = C::kStages, kH = C::kHalves, kN = din_chunks(D);
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    unsigned char *smA = base, *smB = smA + C::kABufs * C::kABytes, *smOut = smB + kS * C::kChunkBytes, *smOne = smOut + C::kStageOut;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smOne + C::kOnesBytes);
    uint64_t *b_full = bars, *b_empty = bars + kS, *a_full = b_empty + kS, *a_empty = a_full + 2, *o_full = a_empty + 2, *o_empty = o_full + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(o_empty + 2);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kS; ++s) mbar_init(smem_u32(b_full + s), 1), mbar_init(smem_u32(b_empty + s), 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(a_full + b), C::kExpandWarps), mbar_init(smem_u32(a_empty + b), 1);
            mbar_init(smem_u32(o_full + b), 1), mbar_init(smem_u32(o_empty + b), C::kOutWarps);
        }
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // rows of 16 elements in two 16-byte columns, 2048 bytes apart: 1 1 1 0 0 0 0 0 | 0 ...
    for (int i = tid; i < C::kOnesBytes / 16; i += C::kThreads)
        reinterpret_cast<uint4 *>(smOne)[i] = i < 128 ? make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async();
    if (warp == C::kMmaWarp) tmem_alloc(smem_u32(tmem_slot), 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (!p.sl.late) grid_dep_wait();
    grid_dep_launch();

    const int tile0 = p.tile0 + (int)((int64_t)p.n_tiles * blockIdx.x / gridDim.x), tile1 = p.tile0 + (int)((int64_t)p.n_tiles * (blockIdx.x + 1) / gridDim.x);
    auto tile_of = [&](int tile) { return key_tile<kDinBlock, false>(p.sl, tile, p.mini_batch); };
    auto req_of = [&](int tile) { return p.sl.tiles ? p.sl.tiles[tile].req - p.req0 : 0; };   // (a single request has no table)

    if (warp < C::kOutWarps) {
        // ===================== rows out =====================
        constexpr int kCols = kDinCols * 4 / C::kOutWarps;   // columns of an item per warp
        const int wq = warp & 3, row = wq * 32 + lane, col0 = (warp >> 2) * kCols;
        const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
        unsigned char *stg = smOut + warp * C::kSlabs * 2048;
        uint32_t slab = 0, it = 0;
        bool ok = true;
        for (int tile = tile0; ok && tile < tile1; ++tile) {
            const KeyTile t = tile_of(tile);
            bool good = false;
            if (row < t.cnt && t.L > 0) {
                const int id = p.sl.ids[t.pos0 + row];
                good = id >= 0 && (int64_t)id < p.M;
            }
            const float scale = (0.5f / (float)D) * (p.din_mean ? 1.0f / (float)t.L : 1.0f);
            const bool whole = wq * 32 + 32 <= t.cnt;
            const uint2 *flags = reinterpret_cast<const uint2 *>(p.image + (size_t)req_of(tile) * din_image_step(D) + din_image_bytes(D));
            for (int half = 0; half < kH; ++half, ++it) {
                const int b = (int)(it & 1u);
                uint32_t infinite = 0u;
#pragma unroll
                for (int c0 = 0; c0 < kCols; c0 += 32) infinite |= __ldcg(&flags[(half * kDinCols + col0 + c0) >> 5].x);
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(o_full + b), (it >> 1) & 1u, abort_flag)))) break;
                tc_fence_after();
#pragma unroll 1
                for (int c0 = col0; c0 < col0 + kCols; c0 += 32) {
                    uint32_t r[32], packed[16];
                    tmem_ld32(lane_base + (uint32_t)(b * kDinCols + c0), r);
                    tmem_ld_wait();
                    if (c0 + 32 == col0 + kCols) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(o_empty + b));
                    }
                    if (infinite) {
                        const uint2 f = __ldcg(&flags[(half * kDinCols + c0) >> 5]);
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if ((f.x >> i) & 1u) r[i] = __float_as_uint(__uint_as_float(r[i]) * __uint_as_float(0x7F800000u | ((f.y >> i) & 1u) << 31));
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const __nv_bfloat162 h = __floats2bfloat162_rn(good ? __uint_as_float(r[2 * i]) * scale : 0.f, good ? __uint_as_float(r[2 * i + 1]) * scale : 0.f);
                        packed[i] = *reinterpret_cast<const uint32_t *>(&h);
                    }
                    const int col = p.x_din + half * kDinCols + c0;
                    if (whole) {   // 32 rows x 32 columns through a 64-byte swizzled slab and an asynchronous tile store
                        unsigned char *sb = stg + slab * 2048;
                        if (lane == 0) bulk_wait_read<C::kSlabs - 1>();
                        __syncwarp();
                        const int swz = (lane >> 1) & 3;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            *reinterpret_cast<uint4 *>(sb + lane * 64 + ((q ^ swz) << 4)) = make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2], packed[4 * q + 3]);
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(&tmapX, smem_u32(sb), col, (int)(t.pos0 + wq * 32));
                            bulk_commit();
                        }
                        slab ^= 1u;
                    } else if (row < t.cnt) {
                        uint4 *dst = reinterpret_cast<uint4 *>(p.X + (size_t)(t.pos0 + row) * p.x_stride + col);
#pragma unroll
                        for (int q = 0; q < 4; ++q) dst[q] = make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2], packed[4 * q + 3]);
                    }
                }
            }
        }
        if (lane == 0) bulk_wait<0>();
    } else if (warp == C::kMmaWarp) {
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(kTcTile, kDinCols);
            uint64_t ones = umma_desc_sw128(smem_u32(smOne));   // without swizzle: 16-byte columns 2048 bytes apart, 8-row groups 128
            ones = (ones & ~((uint64_t)7 << 61) & ~((uint64_t)0x3FFF << 32)) | ((uint64_t)(128u >> 4) << 32) | ((uint64_t)(2048u >> 4) << 16);
            uint32_t it = 0, chunk = 0;   // chunk: chunks so far (d = 256), requests so far (d = 128)
            int k = 0, req = tile0 < tile1 ? req_of(tile0) : -1;
            bool ok = true, fresh = true;
            for (int tile = tile0; ok && tile < tile1; ++tile, ++k) {
                const int ab = k & 1, req_next = tile + 1 < tile1 ? req_of(tile + 1) : -1;
                if (!(ok = mbar_wait(smem_u32(a_full + ab), (uint32_t)((k >> 1) & 1), abort_flag))) break;
                if (C::kResident && fresh && !(ok = mbar_wait(smem_u32(b_full), chunk & 1u, abort_flag))) break;
                const uint64_t a = umma_desc_sw128(smem_u32(smA + ab * C::kABytes));
                for (int half = 0; ok && half < kH; ++half, ++it) {
                    const int b = (int)(it & 1u);
                    if (it >= 2 && !(ok = mbar_wait(smem_u32(o_empty + b), ((it - 2) >> 1) & 1u, abort_flag))) break;
                    tc_fence_after();
#pragma unroll
                    for (int n = 0; n < kN; ++n) {
                        int s = n;
                        if (!C::kResident) {
                            s = (int)(chunk % kS);
                            if (!(ok = mbar_wait(smem_u32(b_full + s), (chunk / kS) & 1u, abort_flag))) break;
                            tc_fence_after();
                        }
                        const uint64_t bd = umma_desc_sw128(smem_u32(smB + s * C::kChunkBytes));
                        if (n < kN - 1) {
                            const uint64_t ad = a + (uint64_t)(uint32_t)((n % (D / 64)) * (16384 >> 4));
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                umma_bf16(tmem_base + (uint32_t)(b * kDinCols), ad + (uint64_t)(2 * kk), bd + (uint64_t)(2 * kk), idesc, n > 0 || kk > 0 ? 1u : 0u);
                        } else
                            umma_bf16(tmem_base + (uint32_t)(b * kDinCols), ones, bd, idesc, 1u);
                        if (!C::kResident) umma_commit(smem_u32(b_empty + s)), ++chunk;
                    }
                    if (!ok) break;
                    umma_commit(smem_u32(o_full + b));
                    if (half == kH - 1) umma_commit(smem_u32(a_empty + ab));
                }
                fresh = req_next != req;
                req = req_next;
                if (C::kResident && ok && fresh) umma_commit(smem_u32(b_empty)), ++chunk;   // the request's last product
            }
        }
        __syncwarp();
    } else if (warp == C::kLoadWarp) {
        if (lane == 0) {
            uint32_t chunk = 0;
            bool ok = true;
            int req = -1, req_next = tile0 < tile1 ? req_of(tile0) : 0;
            for (int tile = tile0; ok && tile < tile1; ++tile) {
                const bool fresh = req_next != req;
                req = req_next;
                if (tile + 1 < tile1) req_next = req_of(tile + 1);   // a tile ahead of its use
                const unsigned char *image = p.image + (size_t)req * din_image_step(D);
                if constexpr (C::kResident) {
                    if (!fresh) continue;
                    if (!(ok = mbar_wait(smem_u32(b_empty), (chunk & 1u) ^ 1u, abort_flag))) break;
                    mbar_expect_tx(smem_u32(b_full), (uint32_t)(kN * C::kChunkBytes));
#pragma unroll 1
                    for (int n = 0; n < kN; ++n) bulk_load(smem_u32(smB + n * C::kChunkBytes), image + (size_t)n * D * 128, (uint32_t)C::kChunkBytes, smem_u32(b_full));
                    ++chunk;
                } else
                for (int half = 0; ok && half < kH; ++half)
                    for (int n = 0; n < kN; ++n, ++chunk) {
                        const int s = (int)(chunk % kS);
                        if (!(ok = mbar_wait(smem_u32(b_empty + s), ((chunk / kS) & 1u) ^ 1u, abort_flag))) break;
                        mbar_expect_tx(smem_u32(b_full + s), (uint32_t)C::kChunkBytes);
                        bulk_load(smem_u32(smB + s * C::kChunkBytes), image + ((size_t)n * D + half * kDinCols) * 128, (uint32_t)C::kChunkBytes, smem_u32(b_full + s));
                    }
            }
        }
        __syncwarp();
    } else {
        // ===================== item signatures -> +-1 in bf16 (256 threads, two per row) =====================
        // ids two tiles ahead of their use, signatures one
        constexpr int kW = D / 128;
        const int i = tid - C::kExpandWarp0 * 32, row = i >> 1, side = i & 1;
        auto id_of = [&](int tile) {
            if (tile >= tile1) return -1;
            const KeyTile t = tile_of(tile);
            const int id = row < t.cnt ? p.sl.ids[t.pos0 + row] : -1;
            return (int64_t)id < p.M ? id : -1;   // an id outside the table: a row of zeros
        };
        auto fetch = [&](int id, uint64_t (&v)[kW]) {
#pragma unroll
            for (int q = 0; q < kW; ++q) v[q] = id >= 0 ? __ldg(reinterpret_cast<const uint64_t *>(p.sig + (size_t)id * (D / 8)) + side * kW + q) : 0ull;
        };
        int k = 0, id = id_of(tile0), id_next = id_of(tile0 + 1);
        uint64_t bits[kW], bits_next[kW];
        fetch(id, bits);
        for (int tile = tile0; tile < tile1; ++tile, ++k) {
            const int ab = k & 1;
            fetch(id_next, bits_next);
            const int id_after = id_of(tile + 2);
            if (k >= 2 && !__all_sync(0xffffffffu, mbar_wait(smem_u32(a_empty + ab), (uint32_t)(((k - 2) >> 1) & 1), abort_flag))) break;
#pragma unroll
            for (int q = 0; q < kW; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    expand_bits32(smA + ab * C::kABytes + (side * kW + q) * 16384 + row * 128, 4 * h, row & 7, (uint32_t)(bits[q] >> (32 * h)), id >= 0 ? 0x3F803F80u : 0u);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(a_full + ab));
            id = id_next, id_next = id_after;
#pragma unroll
            for (int q = 0; q < kW; ++q) bits[q] = bits_next[q];
        }
    }

    if (*abort_flag) {
        if (tid == 0) atomicOr(p.sl.status, AIF_STATUS_TIMEOUT);
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == C::kMmaWarp) tmem_dealloc(tmem_base, 256);
    if (p.sl.late && blockIdx.x == 0) grid_dep_wait();
}

struct DinPlan {
    CUtensorMap tmap_s;
    float4 *records = nullptr;
    unsigned char *image = nullptr;
    int records_cap = 0, requests = 0;
    int at_once[4] = {};   // clusters of 1, 2, 4, 8 CTAs of k_din_sums that the machine holds
};

// CTAs per request, a power of two and a cluster: rounds of clusters times a CTA's key blocks and its start and end (about eight blocks'
// worth).  Of clusters of eight the machine may hold fewer than 148 / 8: sixteen at a time took two rounds.
int din_parts(const DinPlan &pl, int n_req, int d, int max_L)
{
    const int blocks = (max_L + kDinBlock - 1) / kDinBlock, clusters = n_req * (d / kDinCols);
    int best = 1;
    int64_t least = 0;
    for (int i = 0; i < 4; ++i) {
        const int parts = 1 << i;
        if (pl.at_once[i] < 1 || (parts > 1 && (parts > blocks || parts * clusters > pl.records_cap))) continue;
        const int64_t cost = (int64_t)((clusters + pl.at_once[i] - 1) / pl.at_once[i]) * ((blocks + parts - 1) / parts + 8);
        if (i == 0 || cost < least) best = parts, least = cost;
    }
    return best;
}

// A launch's work in key blocks of 128: of its tiles, and of its requests, each with eight blocks' worth of start and end.
struct DinWork {
    int64_t tile_blocks = 0, request_blocks = 0;
    int requests = 0;
    void add(int64_t tiles, int L)
    {
        const int64_t b = ((int64_t)L + kDinBlock - 1) / kDinBlock;
        tile_blocks += tiles * b, request_blocks += b + 8, requests += 1;
    }
};

// The sums save of every tile's pass over the keys what the product costs there (0.7 us per 148 tiles and block), and cost two launches (about
// 10 us before and behind the others; a round more 25) and a pass over the keys of every request with d output columns, whether the request has one
// tile or a hundred.  This way / the other, us:
// d = 128, LSH-DIN and SimTier: 64 x 5000 candidates of 300 keys 658 / 675 with all blocks on, of 1000 752 / 827; 8 x 5000 of 1000 91.1 / 91.6;
// 1 x 3000 of 10^4 48.5 / 47.2; 8 x 1000 of 6000 57.9 / 60.3; 16 x 500 of 8000 68.8 / 70.0; 32 x 256 of 7000 74.6 / 69.9; 148 x 128 of 4000
// 103 / 83; 256 x 100 of 1500 127 / 103; 1024 x 30 of 400 337 / 192.  One key block each 458 / 447.
// d = 128, LSH-DIN alone: 8 x 1000 of 6000 41.5 / 53.6; 32 x 256 of 7000 52.0 / 62.8; 64 x 128 of 10^4 84.2 / 87.2; 148 x 128 of 4000 87.5 / 80.1.
// d = 256, both: 32 x 2000 of 1000 437 / 423, of 2000 451 / 479; 4 x 4000 of 2000 137 / 137, of 5000 149 / 173; 16 x 500 of 10^4 122 / 123; 32 x 256
// of 10^4 152 / 125; 148 x 128 of 4200 247 / 160.  LSH-DIN alone: 16 x 500 of 10^4 99.4 / 115; 32 x 256 of 10^4 127 / 119.
bool din_pays(const aif_config &c, const DinWork &w, int max_L)
{
    const bool tiers = c.blocks & AIF_BLK_SIMTIER;
    const int blocks = (max_L + kDinBlock - 1) / kDinBlock, rounds = (w.requests + kDinRequests - 1) / kDinRequests;
    const int64_t tiles = w.tile_blocks - 5500ll * (rounds - 1);
    if (c.d == 128) return blocks >= 3 && w.tile_blocks >= 148 * 20 && 10 * tiles - (tiers ? 13 : 8) * w.request_blocks >= (tiers ? 23700 : 4000);
    return blocks >= 8 && w.tile_blocks >= 148 * 32 && 10 * tiles >= (tiers ? 35 : 22) * w.request_blocks;
}

}  // namespace

bool tc_din_supported(const aif_config &c)
{
    return c.dtype == AIF_BF16 && (c.blocks & AIF_BLK_LSH_DIN) && (c.d == 128 || c.d == 256) && c.lsh_bits == c.d && c.n_categories == 0 && encode_fn() != nullptr;
}

// Scratch for the requests of a round; without room for it the context does with the pass over the pairs.
cudaError_t tc_din_prepare(aif_ctx *ctx)
{
    const aif_config &c = ctx->cfg;
    DinWork most;
    most.add((int64_t)tc_tile_capacity(ctx), c.L_max);
    if (!din_pays(c, most, c.L_max)) return cudaSuccess;   // no launch of this context is large enough
    const int requests = c.max_user_states < kDinRequests ? c.max_user_states : kDinRequests;
    const size_t n = (size_t)requests * (c.d / kDinCols), records = n < 148 ? 148 : n;   // din_parts: more than one part only within them
    const size_t rec_bytes = records * din_record_bytes(c.d), image_bytes = (size_t)requests * din_image_step(c.d);
    void *rec = nullptr, *image = nullptr;
    if (cudaMalloc(&rec, rec_bytes) != cudaSuccess || cudaMalloc(&image, image_bytes) != cudaSuccess) {
        if (rec) cudaFree(rec);
        cudaGetLastError();
        return cudaSuccess;
    }
    ctx->allocations.push_back(rec), ctx->allocations.push_back(image);
    ctx->device_bytes += (int64_t)(rec_bytes + image_bytes);
    DinPlan *pl = new DinPlan();
    ctx->tc_din_plan = pl;
    pl->records = (float4 *)rec, pl->image = (unsigned char *)image, pl->records_cap = (int)records, pl->requests = requests;
    const cuuint64_t dims[3] = {(cuuint64_t)c.d, (cuuint64_t)c.L_max, (cuuint64_t)c.max_user_states};
    const cuuint64_t strides[2] = {(cuuint64_t)c.d * 2, (cuuint64_t)ctx->slot_bytes};
    const cuuint32_t box[3] = {64, kDinBlock, 1}, estr[3] = {1, 1, 1};
    if (encode_fn()(&pl->tmap_s, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ctx->slots[0].dev.S), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    auto allow = [](auto kernel, size_t smem) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); };
    auto clusters = [&](auto kernel, int threads, size_t smem) {
        for (int i = 0; i < 4; ++i) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(1u << i), cfg.blockDim = dim3((unsigned)threads), cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = 1u << i, attr.val.clusterDim.y = 1, attr.val.clusterDim.z = 1;
            cfg.attrs = &attr, cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&pl->at_once[i], kernel, &cfg) != cudaSuccess) cudaGetLastError(), pl->at_once[i] = i == 0 ? 148 : 0;
        }
    };
    cudaError_t e;
    if (c.d == 128) {
        e = allow(k_din_sums<128>, DinSumsCfg<128>::kSmem);
        if (e == cudaSuccess) e = allow(k_din_apply<128>, DinApplyCfg<128>::kSmem);
        clusters(k_din_sums<128>, DinSumsCfg<128>::kThreads, DinSumsCfg<128>::kSmem);
    } else {
        e = allow(k_din_sums<256>, DinSumsCfg<256>::kSmem);
        if (e == cudaSuccess) e = allow(k_din_apply<256>, DinApplyCfg<256>::kSmem);
        clusters(k_din_sums<256>, DinSumsCfg<256>::kThreads, DinSumsCfg<256>::kSmem);
    }
    return e;
}

void tc_din_destroy(aif_ctx *ctx)
{
    delete reinterpret_cast<DinPlan *>(ctx->tc_din_plan);
    ctx->tc_din_plan = nullptr;
}

bool tc_din_pays(const aif_ctx *ctx, const ScoreLaunch &sl)
{
    const aif_config &c = ctx->cfg;
    const DinPlan *pl = reinterpret_cast<const DinPlan *>(ctx->tc_din_plan);
    if (!pl || sl.grouped) return false;
    DinWork w;
    for (int r = 0; r < sl.n_req; ++r) {
        const ReqDev &rq = sl.reqs_host ? sl.reqs_host[r] : sl.single;
        w.add(tiles_of(rq.n, kTcTile, c.mini_batch), ctx->slots[(size_t)rq.slot].L);
    }
    return din_pays(c, w, sl.max_L);
}

int din_requests_at_once(const aif_ctx *ctx) { return reinterpret_cast<const DinPlan *>(ctx->tc_din_plan)->requests; }

static int round_of(const DinPlan &pl, const ScoreLaunch &sl, int r0) { return sl.n_req - r0 < pl.requests ? sl.n_req - r0 : pl.requests; }

cudaError_t launch_din_sums(const aif_ctx *ctx, const ScoreLaunch &sl, int r0, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    const DinPlan *pl = reinterpret_cast<const DinPlan *>(ctx->tc_din_plan);
    DinSums p{};
    const int n_req = round_of(*pl, sl, r0);
    p.slots = sl.slots, p.reqs = sl.reqs ? sl.reqs + r0 : nullptr, p.single = sl.single, p.late = sl.late, p.status = sl.status;
    p.parts = din_parts(*pl, n_req, c.d, sl.max_L), p.records = pl->records, p.image = pl->image;
    if ((int64_t)p.parts * n_req * (c.d / kDinCols) > pl->records_cap) return cudaErrorInvalidValue;
    auto go = [&](auto kernel, int threads, size_t smem) {
        return launch_pdl_cluster(kernel, dim3(p.parts, c.d / kDinCols, n_req), dim3(threads), smem, (unsigned)p.parts, st, pl->tmap_s, p);
    };
    const cudaError_t e = c.d == 128 ? go(k_din_sums<128>, DinSumsCfg<128>::kThreads, DinSumsCfg<128>::kSmem)
                                     : go(k_din_sums<256>, DinSumsCfg<256>::kThreads, DinSumsCfg<256>::kSmem);
    count_launch();
    return e;
}

// LSH-DIN rows into columns [x_din, x_din + d) of X, after launch_din_sums of the same round.
cudaError_t launch_din_apply(const aif_ctx *ctx, const ScoreLaunch &sl, int r0, cudaStream_t st, void *X, int x_stride, size_t x_rows, int x_din)
{
    const aif_config &c = ctx->cfg;
    const DinPlan *pl = reinterpret_cast<const DinPlan *>(ctx->tc_din_plan);
    CUtensorMap tmap_x;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)x_stride, (cuuint64_t)x_rows};
        const cuuint64_t strides[1] = {(cuuint64_t)x_stride * 2};
        const cuuint32_t box[2] = {32, 32}, estr[2] = {1, 1};
        if (encode_fn()(&tmap_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, X, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    DinApply p{};
    p.sl = sl, p.sig = ctx->sig, p.image = pl->image, p.M = c.M, p.mini_batch = c.mini_batch;
    p.x_stride = x_stride, p.x_din = x_din, p.din_mean = c.lsh_din_norm == AIF_NORM_MEAN, p.X = (__nv_bfloat16 *)X;
    const int r1 = r0 + round_of(*pl, sl, r0);
    p.req0 = r0, p.tile0 = r0 > 0 ? sl.reqs_host[r0].tile_begin : 0, p.n_tiles = (r1 < sl.n_req ? sl.reqs_host[r1].tile_begin : sl.n_tiles) - p.tile0;
    if (p.n_tiles == 0) return cudaSuccess;   // requests without candidates
    const int grid = p.n_tiles < 148 ? p.n_tiles : 148;
    const cudaError_t e = c.d == 128 ? launch_pdl(k_din_apply<128>, dim3(grid), dim3(DinApplyCfg<128>::kThreads), DinApplyCfg<128>::kSmem, st, tmap_x, p)
                                     : launch_pdl(k_din_apply<256>, dim3(grid), dim3(DinApplyCfg<256>::kThreads), DinApplyCfg<256>::kSmem, st, tmap_x, p);
    count_launch();
    return e;
}

}  // namespace aif
