// SimTier on the tensor cores (sm_100a; Section 4.2, eqs. 6 and 9) for tiles of 128 candidates against the request's behaviour
// sequence: up to eight tiers, without the product of eq. 8 (whose rows come from aif_tc_din.cu, or with the counts from aif_tc_lsh.cu).
//
// The match counts are a +-1 product as in aif_tc_lsh.cu, but what a pair costs outside the tensor cores is what bounds the
// kernel, so the product does as much of the tier arithmetic as it can and the rest is bit-sliced:
//   * The accumulator is fp16 (one value per 32-bit column; a packing load puts two columns into a register): every instruction on
//     scores works on two pairs.
//   * One more product step of K = 32 adds a constant: the accumulator holds (2 matches + delta) 2^-9.  With delta between
//     -2 d' / N * 1/2 and the next value that a pair can take, round-to-nearest of (2 matches + delta) N / (2 d') is
//     floor(matches N / d') for every possible count (host check in tier_offset); the item's bits are +-2^-9, the sequence's +-1.
//   * One fp16 multiply-add then leaves tier + 1 as a subnormal, 2^-24 units, which is the integer itself in the register: no
//     masks, no shifts.  (The + 1 keeps a rounded negative from becoming minus zero, whose sign bit is not an integer's.)
//   * Two more multiply-adds and an integer one gather four pairs into the nibbles of a byte permute's selector; the permute
//     looks up four bytes with one bit per tier.  The last tier, and matches = d', have a nibble of 8 or 9: the permute answers
//     with the sign of a table byte, zero; the last tier is the rest of the total.
//   * The bytes are summed bit-sliced: eight words hold the binary digits of 32 counters (7 tiers x 4 byte positions), a carry-save
//     adder (two three-input logic instructions) takes in two words, halving with every digit.  The digits are transposed into bytes and
//     added to 32-bit counters when the tile ends.
// Per pair 2.1 instructions (2.9 with everything around the loop), on two half-rate pipes (integer, and the fp16 half of the FMA pipe) in equal
// shares, against 5.0 where the counts also become the operand of eq. 8's product: 592 cycles per 128 keys for 320 of products (means over the SMs,
// 4 requests of 10^4 candidates, 10^4 keys; 16 of them: 215 us; both blocks in one pass over the pairs: 1600 cycles, 650 us).  What bounds it:
// issue slots, 0.62 of them taken.
// Tried: sixteen warps over two buffers of 256 columns with one issuing lane (673 cycles, the lane), twelve warps with all 128 columns of a unit
// in registers (617 to 640: three warps to a scheduler do not cover each other's waits of 200 cycles for scores and 200 for their load), the
// counters emptied every seven units (490 cycles of a warp each time; now carried into eight more digits), 32 columns at a time with the next ones
// on their way (432 us for the whole call, 425 so: the registers).
//
// One CTA per SM walks over the tiles (or pieces) blockIdx.x, blockIdx.x + gridDim.x, ...  Keys go in units of 128.  Warps (640 threads):
//   0-15   tiers of a unit for a quarter of the rows (a thread owns a row); four warps share a quarter and take every fourth unit
//   16 17  one lane each issues the products, of even and of odd units: a wait costs a lane as long as three products take, which the
//          other one's products cover.  Warp 16 allocates tensor memory
//   18     one lane streams the +-1 signatures of the sequence with TMA
//   19     expands the item signatures of the next tile into one of two operand buffers
// Tensor memory: four score buffers of 128 columns.  Every wait is bounded.
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <cmath>
#include <type_traits>

#include "aif_device.cuh"
#include "aif_internal.h"
#include "aif_tc_ptx.cuh"

namespace aif {
namespace {

constexpr int kUnit = 128;       // keys per product
// Binary digits of a bit-sliced counter: eight that every unit works on, and eight that take the carries of eight units at once (a unit
// adds at most 32 to a counter, so eight units carry at most once out of the lower digits).
constexpr int kTierDigits = 8;
constexpr int kTierUnits = 2040;   // units until the sixteen digits are emptied into a thread's 32-bit counters

struct TierParams {
    ScoreLaunch sl;
    const uint8_t *sig;      // item signatures [M x D / 8], first bit = most significant bit of byte 0
    int64_t M;
    int32_t mini_batch;
    int32_t x_stride;        // elements per row of X
    int32_t x_tier;          // first SimTier column of X (64 columns, the first n_tiers used)
    int32_t n_tiers;         // at most 8
    int32_t tier_mean;       // divide by the sequence length
    uint32_t bias;           // four E4M3 values whose sum times 2^-3 is (2 matches + delta) 2^-9 of a pair without any product
    uint32_t scale;          // fp16 pair: tier in units of 2^-24 per accumulator unit
    __nv_bfloat16 *X;
};

template <int D>
struct TierCfg {
    static constexpr int kBlock = D <= 128 ? 128 : 64;   // keys per block of the launch's pieces (key_tile)
    static constexpr int kQChunks = D / 128;
    static constexpr int kQBytes = kQChunks * 128 * 128;
    static constexpr int kGChunkBytes = kUnit * 128;
    static constexpr int kGBytes = kQChunks * kGChunkBytes;
    static constexpr int kScores = 4;                    // score buffers in tensor memory, one per counting warp of a quarter
    // Unit u: buffer, barrier and counting warp u mod 4, issuer u mod 2.  (A barrier's phases must be met one by one by whoever waits on it:
    // a parity wait is also answered by the phase before last.)  As many stages of the key ring: the keys of a unit are never announced on
    // its barrier before that has done with the unit four before it.
    static constexpr int kStages = 4;
    static constexpr int kBiasBytes = (128 + kUnit) * 32;
    static constexpr int kShare = kScores;               // warps per quarter of the rows
    static constexpr int kConvWarps = 4 * kShare, kMmaWarp = kConvWarps, kTmaWarp = kConvWarps + 2;
    static constexpr int kThreads = 20 * 32;
    static constexpr int kCountBytes = 2 * (kShare - 1) * 8 * 128 * 4;   // [tile parity][warps of the quarter but the first][7 tiers, totals][row]
    static constexpr size_t kSmem = 1024 + 2 * kQBytes + kStages * kGBytes + kBiasBytes + 512 + kCountBytes;
    static_assert(kSmem <= 227 * 1024, "shared memory");
    static_assert(kStages == kScores && (kStages + 2 * kScores + 5) * 8 + 8 <= 512, "barriers");
};

// 32 lanes x 64 columns, the low halves of two adjacent columns in one register.
__device__ __forceinline__ void tmem_ld64_pack16(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

template <int TABLE>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(a), "r"(b), "r"(c), "n"(TABLE));
    return r;
}
// Full adder on 32 single bits: digit += a + b, the carries returned.
__device__ __forceinline__ uint32_t csa(uint32_t &digit, uint32_t a, uint32_t b)
{
    const uint32_t carry = lop3<0xE8>(digit, a, b);
    digit = lop3<0x96>(digit, a, b);
    return carry;
}

__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<const __half2 *>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<const uint32_t *>(&v); }
__device__ __forceinline__ uint32_t byte_perm(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// 64 scores of a row (two to a register) into the bit-sliced counters' first four digits; the carry into the fifth is returned.
__device__ __forceinline__ uint32_t count_tiers(const uint32_t (&v)[32], __half2 scale, uint32_t (&digit)[kTierDigits])
{
    const __half2 one = as_half2(0x00010001u), sixteen = as_half2(0x4C004C00u);
    uint32_t w[2][2], twos[2], fours[2], eights[2];
#pragma unroll
    for (int i = 0; i < 8; ++i) {   // eight scores each: two words of four
        uint32_t t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) t[q] = as_u32(__hfma2(as_half2(v[4 * i + q]), scale, one));
        const uint32_t lo = as_u32(__hfma2(as_half2(t[1]), sixteen, as_half2(t[0]))), hi = as_u32(__hfma2(as_half2(t[3]), sixteen, as_half2(t[2])));
        const uint32_t sel = hi * 256u + lo;
        w[i & 1][0] = byte_perm(0x04020100u, 0x40201008u, sel), w[i & 1][1] = byte_perm(0x04020100u, 0x40201008u, sel >> 16);
        if (i & 1) {
            twos[0] = csa(digit[0], w[0][0], w[0][1]), twos[1] = csa(digit[0], w[1][0], w[1][1]);
            fours[(i >> 1) & 1] = csa(digit[1], twos[0], twos[1]);
            if ((i & 3) == 3) eights[(i >> 2) & 1] = csa(digit[2], fours[0], fours[1]);
        }
    }
    return csa(digit[3], eights[0], eights[1]);
}
// digit += c from digit FROM on; what is carried out of the last one is returned.
template <int FROM>
__device__ __forceinline__ uint32_t carry_up(uint32_t (&digit)[kTierDigits], uint32_t c)
{
#pragma unroll
    for (int k = FROM; k < kTierDigits; ++k) {
        const uint32_t next = digit[k] & c;
        digit[k] ^= c;
        c = next;
    }
    return c;
}

// Bit-sliced counters -> 32-bit ones: the 8 x 8 bits of every byte position transposed, then the four positions summed.
__device__ __forceinline__ void flush_tiers(uint32_t (&digit)[kTierDigits], uint32_t (&cnt)[7], int shift)
{
    auto swap = [&](uint32_t &a, uint32_t &b, int s, uint32_t m) {
        const uint32_t t = ((a >> s) ^ b) & m;
        b ^= t, a ^= t << s;
    };
#pragma unroll
    for (int k = 0; k < 4; ++k) swap(digit[k], digit[k + 4], 4, 0x0F0F0F0Fu);
#pragma unroll
    for (int k = 0; k < 8; k += 4) swap(digit[k], digit[k + 2], 2, 0x33333333u), swap(digit[k + 1], digit[k + 3], 2, 0x33333333u);
#pragma unroll
    for (int k = 0; k < 8; k += 2) swap(digit[k], digit[k + 1], 1, 0x55555555u);
#pragma unroll
    for (int t = 0; t < 7; ++t) cnt[t] += __dp4a(digit[t], 0x01010101u, 0u) << shift;
#pragma unroll
    for (int k = 0; k < kTierDigits; ++k) digit[k] = 0u;
}

// SPLIT: the launch's tiles are cut into pieces of their keys.
template <int D, bool SPLIT>
__global__ void __launch_bounds__((TierCfg<D>::kThreads), 1) k_tiers(const __grid_constant__ CUtensorMap tmapG, const TierParams p)
{
    using C = TierCfg<D>;
    constexpr int kS = C::kStages, kT = C::kScores;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    unsigned char *smQ = base;
    unsigned char *smG = smQ + 2 * C::kQBytes;
    unsigned char *smBias = smG + kS * C::kGBytes;   // rows of A (128 x 32 bytes), then of B (kUnit x 32 bytes)
    uint64_t *bars = reinterpret_cast<uint64_t *>(smBias + C::kBiasBytes);
    uint64_t *g_empty = bars, *s_full = g_empty + kS, *ready = s_full + kT, *q_full = ready + kT, *q_empty = q_full + 2;
    uint64_t *q_first = q_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(q_first + 1);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    uint32_t *count_s = reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned char *>(bars) + 512);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kS; ++s) mbar_init(smem_u32(g_empty + s), 1);
        // ready: a unit's keys have arrived and its score buffer has been read by its four warps; one wait of an issuer for both
        for (int v = 0; v < kT; ++v) mbar_init(smem_u32(s_full + v), 1), mbar_init(smem_u32(ready + v), 5);
        for (int b = 0; b < 2; ++b) mbar_init(smem_u32(q_full + b), 1), mbar_init(smem_u32(q_empty + b), 2);   // both issuers
        mbar_init(smem_u32(q_first), C::kConvWarps * 32);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the constant step's operands: every 16-byte piece of A's rows is the same, B's rows are all 2^-4 (two pieces of 16 to a row)
    for (int i = tid; i < C::kBiasBytes / 16; i += C::kThreads)
        reinterpret_cast<uint4 *>(smBias)[i] = i < 128 * 2 ? make_uint4(p.bias, 0u, 0u, 0u) : make_uint4(0x18181818u, 0x18181818u, 0x18181818u, 0x18181818u);
    fence_proxy_async();
    if (warp == C::kMmaWarp) tmem_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (!p.sl.late) grid_dep_wait();
    grid_dep_launch();   // (after the wait: see ScoreLaunch::late)

    const int n_tiles = key_jobs<SPLIT>(p.sl);
    auto tile_of = [&](int tile) { return key_tile<C::kBlock, SPLIT>(p.sl, tile, p.mini_batch); };
    auto units_of = [](int L) { return L > kUnit ? (L + kUnit - 1) / kUnit : 1; };   // an empty tile passes through with one

    // Item signatures of N rows (r0, r0 + step, ...) as +-2^-9 bytes in the operand layout (128-byte swizzled K-major chunks): 8
    // threads per row, 16 bits each per 128-bit chunk, all of a thread's signature bytes requested before the first is expanded.
    auto expand_rows = [&](unsigned char *q, int r0, int step, int sub, auto n_const, auto id_of) {
        constexpr int N = decltype(n_const)::value;
        uint16_t two[N][C::kQChunks];
        uint32_t good = 0u;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int id = id_of(i);
            if (id >= 0) good |= 1u << i;
#pragma unroll
            for (int c = 0; c < C::kQChunks; ++c)
                two[i][c] = __ldg(reinterpret_cast<const uint16_t *>(p.sig + (size_t)max(id, 0) * (D / 8) + c * 16 + sub * 2));
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int r = r0 + step * i;
#pragma unroll
            for (int c = 0; c < C::kQChunks; ++c) {
                uint4 v = expand_sig16(two[i][c] & 0xFFu, two[i][c] >> 8);
                auto small = [&](uint32_t x) { return (good >> i) & 1u ? (x & 0x80808080u) | 0x01010101u : 0u; };   // E4M3: +-2^-9
                v = make_uint4(small(v.x), small(v.y), small(v.z), small(v.w));
                *reinterpret_cast<uint4 *>(q + c * 16384 + r * 128 + ((sub ^ (r & 7)) << 4)) = v;
            }
        }
    };

    if (warp < C::kConvWarps) {
        // ===================== tiers =====================
        const int wq = warp & 3, h = warp >> 2;
        const int row = wq * 32 + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
        const uint32_t s_col = lane_base + (uint32_t)(h * kUnit);
        const __half2 scale = as_half2(p.scale);
        if (lane == 0) mbar_arrive(smem_u32(ready + h));   // the buffers are free for the first units
        bool ok = true;
        uint32_t phase = 0;     // of this warp's barriers
        int k = 0, skip = h;    // skip: units until this warp's next one
        if ((int)blockIdx.x < n_tiles) {
            // the CTA's first tile has nobody to prefetch it: these warps build its signature operand
            const KeyTile t = tile_of(blockIdx.x);
            int idv[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = (tid >> 3) + 64 * i;
                idv[i] = r < t.cnt ? p.sl.ids[t.pos0 + r] : -1;
                if ((int64_t)idv[i] >= p.M) idv[i] = -1;
            }
            expand_rows(smQ, tid >> 3, 64, tid & 7, std::integral_constant<int, 2>{}, [&](int i) { return idv[i]; });
            fence_proxy_async();
            mbar_arrive(smem_u32(q_first));
        }
        for (int tile = blockIdx.x; ok && tile < n_tiles; tile += gridDim.x, ++k) {
            const KeyTile t = tile_of(tile);
            uint32_t digit[kTierDigits], upper[kTierDigits], carried = 0u, cnt[7];
#pragma unroll
            for (int i = 0; i < kTierDigits; ++i) digit[i] = upper[i] = 0u;
#pragma unroll
            for (int i = 0; i < 7; ++i) cnt[i] = 0u;
            int n_valid = 0, n_pad = 0, since = 0;
            const int nu = units_of(t.L);
            int u = skip;
            // Keys are counted by 64.  Columns between the end of the sequence and the next multiple of 64 have zero signatures (the user side
            // pads to 128): their matches read d' / 2, and they are taken out at the end.
            auto unit = [&](int here) {
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(s_full + h), phase, abort_flag))) return false;
                phase ^= 1u;
                tc_fence_after();
                // (96 registers to a thread: 64 columns at a time)
                uint32_t v[32], c = 0u, c1 = 0u;
                tmem_ld64_pack16(s_col, v);
                tmem_ld_wait();
                if (here > 0) c = count_tiers(v, scale, digit);
                if (here > 64) {
                    tmem_ld64_pack16(s_col + 64u, v);
                    tmem_ld_wait();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(ready + h));   // for the unit four further
                if (here > 64) c1 = count_tiers(v, scale, digit);
                carried |= carry_up<5>(digit, csa(digit[4], c, c1));
                if ((++since & 7) == 0) {
                    carry_up<0>(upper, carried);
                    carried = 0u;
                    if (since == kTierUnits) flush_tiers(digit, cnt, 0), flush_tiers(upper, cnt, 8), since = 0;
                }
                return true;
            };
            const int whole_units = t.L / kUnit;
            for (; ok && u < whole_units; u += kT) ok = unit(kUnit), n_valid += kUnit;
            if (ok && u < nu) {   // the last one, ragged
                const int here = t.L - u * kUnit;
                ok = unit(here), u += kT, n_valid += here, n_pad = (-here) & 63;
            }
            skip = u - nu;
            if (ok) {
                flush_tiers(digit, cnt, 0);
                if (since >= 8 || carried) {
                    carry_up<0>(upper, carried);
                    flush_tiers(upper, cnt, 8);
                }
            }
            // ---- SimTier columns of the tile (eq. 9): 64 bf16 per row, the first n_tiers used.  The four warps of a row quarter meet
            // here once per tile; a failed wait is carried through the barrier so that all leave together.
            uint32_t *all = count_s + (k & 1) * (C::kShare - 1) * 8 * 128 + row;
            if (h > 0) {
                uint32_t *mine = all + (h - 1) * 8 * 128;
#pragma unroll
                for (int i = 0; i < 7; ++i) mine[i * 128] = cnt[i];
                mine[7 * 128] = (uint32_t)n_valid | ((uint32_t)n_pad << 25);   // (a piece has one ragged end: at most 63)
            }
            if (named_bar_or(1 + wq, 32 * C::kShare, !ok)) {
                ok = false;
                break;
            }
            if (h != 0) continue;
            int total = n_valid, pads = n_pad;
#pragma unroll
            for (int i = 0; i < C::kShare - 1; ++i) {
                const uint32_t v = all[(i * 8 + 7) * 128];
                total += (int)(v & 0x1FFFFFFu), pads += (int)(v >> 25);
#pragma unroll
                for (int tt = 0; tt < 7; ++tt) cnt[tt] += all[(i * 8 + tt) * 128];
            }
            bool good = false;
            if (row < t.cnt && t.L_tile > 0) {
                const int id = p.sl.ids[t.pos0 + row];
                good = id >= 0 && (int64_t)id < p.M;
            }
            const float nrm = p.tier_mean ? 1.0f / (float)t.L_tile : 1.0f;
            const bool whole = !SPLIT || t.n_parts == 1;
            uint32_t outw[4];
            int below = 0;
            float prev = 0.f;
#pragma unroll
            for (int tt = 0; tt < 8; ++tt) {
                int c = tt < 7 ? (int)cnt[tt] : 0;
                if (tt == (p.n_tiers >> 1)) c -= pads;
                if (tt == p.n_tiers - 1) c = total - below;   // the closed last tier
                below += c;
                if (!whole && t.n_parts > 0) __stcg(p.sl.split.tiers + ((size_t)(t.pslot + t.part) * 16 + tt) * 128 + row, c);
                const float f = good && tt < p.n_tiers ? (float)c * nrm : 0.f;
                if (tt & 1) {
                    const __nv_bfloat162 o = __floats2bfloat162_rn(prev, f);
                    outw[tt >> 1] = *reinterpret_cast<const uint32_t *>(&o);
                } else
                    prev = f;
            }
            if (whole && row < t.cnt) {
                uint4 *dst = reinterpret_cast<uint4 *>(p.X + (size_t)(t.pos0 + row) * p.x_stride + p.x_tier);
                dst[0] = make_uint4(outw[0], outw[1], outw[2], outw[3]);
#pragma unroll
                for (int q = 1; q < 8; ++q) dst[q] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    } else if (warp < C::kTmaWarp) {
        // ===================== products =====================
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_e4m3_f16(kTcTile, kUnit);
            const int parity = warp - C::kMmaWarp;
            const uint64_t qdesc0 = umma_desc_sw128(smem_u32(smQ)), gdesc0 = umma_desc_sw128(smem_u32(smG));
            const uint64_t abias = umma_desc_plain(smem_u32(smBias), 2048), bbias = umma_desc_plain(smem_u32(smBias + 4096), kUnit * 16);
            // (indices by counting: a remainder is ten dependent instructions of a lone thread, 60 cycles)
            uint32_t phase = 0;
            int k = 0, v = parity, skip = parity;   // skip: units until this lane's next one
            bool ok = true;
            int nu_next = (int)blockIdx.x < n_tiles ? units_of(tile_of(blockIdx.x).L) : 0;
            for (int tile = blockIdx.x; ok && tile < n_tiles; tile += gridDim.x, ++k) {
                const int nu = nu_next, qb = k & 1;
                const int next = tile + (int)gridDim.x;
                nu_next = next < n_tiles ? units_of(tile_of(next).L) : 0;   // fetched a tile ahead of its use
                ok = k == 0 ? mbar_wait(smem_u32(q_first), 0u, abort_flag) : mbar_wait(smem_u32(q_full + qb), (uint32_t)(((k - 1) >> 1) & 1), abort_flag);
                const uint64_t qd = qdesc0 + (uint64_t)(uint32_t)(qb * (C::kQBytes >> 4));
                int u = skip;
                for (; ok && u < nu; u += 2) {
                    if (!(ok = mbar_wait(smem_u32(ready + v), phase, abort_flag))) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + (uint32_t)(v * kUnit);
                    const uint64_t gd = gdesc0 + (uint64_t)(uint32_t)(v * (C::kGBytes >> 4));
                    umma_e4m3(d_tmem, abias, bbias, idesc, 0u);
#pragma unroll
                    for (int kk = 0; kk < D / 32; ++kk)
                        umma_e4m3(d_tmem, qd + (uint64_t)((kk >> 2) * (16384 >> 4) + 2 * (kk & 3)),
                                  gd + (uint64_t)((kk >> 2) * (C::kGChunkBytes >> 4) + 2 * (kk & 3)), idesc, 1u);
                    umma_commit(smem_u32(s_full + v));
                    umma_commit(smem_u32(g_empty + v));
                    v ^= 2;
                    phase ^= (uint32_t)(v == parity);
                }
                skip = u - nu;
                // this lane's products of the tile, if any (after the wait: no arrival for a later tenant before this one's)
                if (ok) umma_commit(smem_u32(q_empty + qb));
            }
        }
        __syncwarp();
    } else if (warp == C::kTmaWarp) {
        // ===================== signatures of the sequence =====================
        if (lane == 0) {
            uint32_t gu = 0;   // units so far, of all tiles
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < n_tiles; tile += gridDim.x) {
                const KeyTile t = tile_of(tile);
                const int nu = units_of(t.L);
                for (int u = 0; u < nu; ++u, ++gu) {
                    const int s = (int)(gu % kS);
                    const uint32_t bar = smem_u32(ready + s);
                    if (!(ok = mbar_wait(smem_u32(g_empty + s), ((gu / kS) & 1u) ^ 1u, abort_flag))) break;
                    mbar_expect_tx(bar, (uint32_t)C::kGBytes);
#pragma unroll
                    for (int c = 0; c < C::kQChunks; ++c)
                        tma_load_3d(smem_u32(smG + s * C::kGBytes + c * C::kGChunkBytes), &tmapG, bar, c * 128, t.key0 + u * kUnit, t.slot);
                }
            }
        }
        __syncwarp();
    } else {
        // ===================== signature operand of the next tile (32 threads) =====================
        const int sub = lane & 7, r0 = lane >> 3;
        int k = 1;
        for (int tile = blockIdx.x + gridDim.x; tile < n_tiles; tile += gridDim.x, ++k) {
            const int qb = k & 1;
            if (k >= 2 && !__all_sync(0xffffffffu, mbar_wait(smem_u32(q_empty + qb), (uint32_t)(((k - 2) >> 1) & 1), abort_flag))) break;
            const KeyTile t = tile_of(tile);
            int idv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = lane + 32 * u;
                int id = r < t.cnt ? p.sl.ids[t.pos0 + r] : -1;
                if ((int64_t)id >= p.M) id = -1;
                idv[u] = id;
            }
#pragma unroll
            for (int half = 0; half < 2; ++half)   // (16 rows at a time: the loads of 32 do not fit in registers)
                expand_rows(smQ + qb * C::kQBytes, r0 + 64 * half, 4, sub, std::integral_constant<int, 16>{},
                            [&](int i) { return __shfl_sync(0xffffffffu, idv[2 * half + (i >> 3)], r0 + 4 * (i & 7)); });
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(q_full + qb));
        }
    }

    if (*abort_flag) {
        if (tid == 0) atomicOr(p.sl.status, AIF_STATUS_TIMEOUT);
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == C::kMmaWarp) tmem_dealloc(tmem_base, 512);
    if (p.sl.late && blockIdx.x == 0) grid_dep_wait();
}

// What the product adds to every pair: delta such that (2 m + delta) N / (2 d') rounds to floor(m N / d') for m = 0 .. d', never from
// a tie, every 2 m + delta (and every partial sum) exact in fp16, and 2^-9 of delta + d' a sum of four E4M3 values times 2^-3.
bool tier_offset(int d, int n_tiers, uint32_t *bias)
{
    for (int frac = 1; frac <= 4; frac *= 2)
        for (int i = -d * frac; i <= 0; ++i) {
            const double delta = (double)i / frac;
            bool good = true;
            for (int m = 0; good && m <= d; ++m) {
                const double x = 2 * m + delta, v = x * n_tiers / (2.0 * d), r = std::floor(v + 0.5);
                good = r == (double)(m * n_tiers / d) && std::fabs(std::fabs(v - r) - 0.5) > 1e-9 && std::fabs(x) * frac <= 2048.0;
            }
            if (!good) continue;
            double rest = (delta + d) / 64.0;
            uint32_t bytes = 0;
            for (int q = 0; q < 4; ++q) {
                const __nv_fp8_e4m3 e((float)rest);
                bytes |= (uint32_t)e.__x << (8 * q);
                rest -= (double)(float)e;
            }
            if (rest != 0.0) continue;
            *bias = bytes;
            return true;
        }
    return false;
}

struct TierPlan {
    CUtensorMap tmap_g, tmap_gg;   // +-1 signatures of the sequences; categories on: of the grouped sequences
    uint32_t bias = 0, scale = 0;
};

}  // namespace

bool tc_tiers_supported(const aif_config &c)
{
    uint32_t bias;
    return c.dtype == AIF_BF16 && (c.blocks & AIF_BLK_SIMTIER) && (c.d == 128 || c.d == 256) && c.lsh_bits == c.d && c.n_tiers >= 1 && c.n_tiers <= 8 &&
           tier_offset(c.d, c.n_tiers, &bias) && encode_fn() != nullptr;
}

cudaError_t tc_tiers_prepare(aif_ctx *ctx)
{
    const aif_config &c = ctx->cfg;
    TierPlan *pl = new TierPlan();
    ctx->tc_tier_plan = pl;
    if (!tier_offset(c.d, c.n_tiers, &pl->bias)) return cudaErrorInvalidValue;
    // tier = (2 m + delta) N / (2 d'): the accumulator holds 2^-9 of the first factor, the result is to have units of 2^-24
    const uint32_t sub = (uint32_t)(c.n_tiers * 256 / c.d);   // N 2^-24 2^9 / (2 d') in units of 2^-24: N 256 / d'
    pl->scale = sub | sub << 16;
    auto encode = [&](CUtensorMap *m, const uint8_t *base, size_t rows) {
        const cuuint64_t dims[3] = {(cuuint64_t)c.lsh_bits, (cuuint64_t)rows, (cuuint64_t)c.max_user_states};
        const cuuint64_t strides[2] = {(cuuint64_t)c.lsh_bits, (cuuint64_t)ctx->slot_bytes};
        const cuuint32_t box[3] = {128, (cuuint32_t)kUnit, 1}, estr[3] = {1, 1, 1};
        return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    if (!encode(&pl->tmap_g, ctx->slots[0].dev.sigE, (size_t)c.L_max)) return cudaErrorInvalidValue;
    if (c.n_categories > 0 && !encode(&pl->tmap_gg, ctx->slots[0].dev.sigEg, ctx->grouped_rows)) return cudaErrorInvalidValue;
    auto allow = [](auto kernel, size_t smem) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); };
    cudaError_t e;
    if (c.d == 128) {
        e = allow(k_tiers<128, false>, TierCfg<128>::kSmem);
        if (e == cudaSuccess) e = allow(k_tiers<128, true>, TierCfg<128>::kSmem);
    } else {
        e = allow(k_tiers<256, false>, TierCfg<256>::kSmem);
        if (e == cudaSuccess) e = allow(k_tiers<256, true>, TierCfg<256>::kSmem);
    }
    return e;
}

void tc_tiers_destroy(aif_ctx *ctx)
{
    delete reinterpret_cast<TierPlan *>(ctx->tc_tier_plan);
    ctx->tc_tier_plan = nullptr;
}

// SimTier rows into columns [x_tier, x_tier + 64) of X.
cudaError_t launch_tiers(const aif_ctx *ctx, const ScoreLaunch &sl, cudaStream_t st, void *X, int x_stride, int x_tier, JoinParams &j)
{
    const aif_config &c = ctx->cfg;
    const TierPlan *pl = reinterpret_cast<const TierPlan *>(ctx->tc_tier_plan);
    TierParams p{};
    p.sl = sl, p.sig = ctx->sig, p.M = c.M, p.mini_batch = c.mini_batch;
    p.x_stride = x_stride, p.x_tier = x_tier, p.n_tiers = c.n_tiers, p.X = (__nv_bfloat16 *)X;
    p.tier_mean = c.simtier_norm == AIF_NORM_MEAN, p.bias = pl->bias, p.scale = pl->scale;
    const bool split = sl.jobs || sl.parts > 1;
    const int jobs = sl.jobs ? sl.n_jobs : sl.n_tiles * (split ? sl.parts : 1), grid = jobs > 148 ? 148 : jobs;
    const CUtensorMap &tg = sl.grouped ? pl->tmap_gg : pl->tmap_g;
    auto go = [&](auto kernel, size_t smem) { return launch_pdl(kernel, dim3(grid), dim3(TierCfg<128>::kThreads), smem, st, tg, p); };
    cudaError_t e;
    if (c.d == 128) e = split ? go(k_tiers<128, true>, TierCfg<128>::kSmem) : go(k_tiers<128, false>, TierCfg<128>::kSmem);
    else e = split ? go(k_tiers<256, true>, TierCfg<256>::kSmem) : go(k_tiers<256, false>, TierCfg<256>::kSmem);
    count_launch();
    j = JoinParams{};
    if (e != cudaSuccess || !split) return e;
    j.sl = sl, j.X = (__nv_bfloat16 *)X, j.M = c.M, j.x_stride = x_stride, j.col = -1, j.x_tier = x_tier, j.n_tiers = c.n_tiers, j.d = c.d;
    j.mini_batch = c.mini_batch, j.tier_mean = p.tier_mean;
    return cudaSuccess;
}

}  // namespace aif
