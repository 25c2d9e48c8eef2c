// Tensor-core scoring path for sm_100a (bf16 storage): the scoring MLP as tcgen05 GEMMs with a fused gather
// prologue and fused epilogues.
//
// One layer = one persistent kernel (k_layer_pair).  A work item is a pair of 128-candidate tiles, one per CTA of a cluster of
// two, times a slice of up to 256 of the layer's outputs.  Roles inside a CTA:
//   epilogue   8 warps: read the fp32 accumulator from TMEM (tcgen05.ld), add the bias (for the first layer the request's
//              cached user partial p_u), ReLU, then either store bf16 activations for the next layer (through a staging slab
//              and a TMA tile store), reduce against w_out and write the logit, or (item side of the nearline pipeline)
//              store without ReLU / pack the sign bits of the outputs
//   MMA        one warp allocates TMEM; one lane of the even CTA issues tcgen05.mma.cta_group::2 (M=256, N<=256, K=16, bf16
//              in, fp32 accumulate)
//   A producer 6 warps: bring the tile's input rows chunk by chunk (64 columns = 128 bytes per row) into the 128B-swizzled
//              K-major layout the MMA reads: with 16-byte cp.async item-table rows by candidate id and cross-feature rows by
//              (field, bucket) from the request's pre-cache, the bucket looked up in the table k_cross_buckets wrote; dense
//              rows (attention output, previous activations, raw item features) by position as one TMA tile per chunk
//   B producer one lane streams the CTA's half of the weight slice with TMA (cp.async.bulk.tensor, 128B swizzle)
// A shared-memory ring (mbarriers) decouples producers from the MMA; two TMEM accumulators of 256 columns alternate so that the
// epilogue of one item overlaps the main loop of the next.  Every wait is bounded: on expiry the CTA raises
// AIF_STATUS_TIMEOUT, all roles leave their loops, TMEM is freed and the kernel returns.
#include <cuda.h>

#include "aif_device.cuh"
#include "aif_internal.h"
#include "aif_tc_ptx.cuh"

namespace aif {
namespace {

constexpr int kABytes = kTcTile * 128;    // one A chunk of one tile: 128 rows x 64 bf16
constexpr int kMaxChunks = 64;
constexpr int kFusedMaxTiles = 148;

enum { SRC_ITEM = 0, SRC_DENSE = 1, SRC_CROSS = 2 };
enum { EPI_STORE = 0, EPI_DOT = 1, EPI_SIGN = 2 };

struct ChunkSrc {
    int32_t kind;
    int32_t off;   // ITEM / DENSE: byte offset inside the source row; CROSS: first cross column of the chunk
};

struct LayerParams {
    ScoreLaunch sl;
    int32_t n_nchunks, n_cols, n_k, mini_batch;
    int32_t n_out;                // outputs of the layer (the last slice may be narrower than n_cols)
    // A sources
    const uint8_t *E;
    int64_t M;
    int32_t e_row_bytes;
    const uint8_t *X;             // dense rows, indexed by candidate position in the launch
    const uint16_t *xb;           // cross-feature buckets [positions x F], written by k_cross_buckets
    const uint8_t *T0;            // cross pre-cache of slot 0; slot i's lies i * slot_bytes further
    int64_t slot_bytes;
    int32_t F, B, dc;
    int32_t check_ids;            // first layer: flag ids outside the table
    // epilogue
    int32_t epi, bias_from_slot, emit_sigmoid, out_stride;
    int32_t linear_out;           // EPI_STORE without the ReLU (output layer of the item-side tower)
    uint8_t *sig_out;             // EPI_SIGN: [positions x out_stride / 8] packed sign bits of the outputs
    const float *bias;
    __nv_bfloat16 *out;           // EPI_STORE: [positions x out_stride]
    const __nv_bfloat16 *w_out;
    const float *b_out;
    ChunkSrc src[kMaxChunks];
};

struct TileInfo {
    ReqDev rq;
    int start, cnt;
    int64_t pos0;   // position of the tile's first candidate in the launch (ids / logits / dense rows)
};

__device__ __forceinline__ TileInfo decode_tile(const LayerParams &p, int tile, int n_tiles)
{
    TileInfo t;
    if (tile >= n_tiles) {   // the second tile of the last group may not exist
        t.rq = ReqDev{0, 0, 0, 0, 0};
        t.start = 0, t.cnt = 0, t.pos0 = 0;
        return t;
    }
    if (p.sl.tiles) {   // looked up once per launch
        const int4 v = *reinterpret_cast<const int4 *>(p.sl.tiles + tile);   // slot, cnt, pos0
        t.rq = ReqDev{v.x, 0, 0, 0, 0};
        t.start = 0, t.cnt = v.y;
        t.pos0 = ((int64_t)(uint32_t)v.w << 32) | (int64_t)(uint32_t)v.z;
        return t;
    }
    t.rq = find_request(p.sl, tile);
    tile_range(tile - t.rq.tile_begin, t.rq.n, kTcTile, p.mini_batch, t.start, t.cnt);
    t.pos0 = t.rq.off + t.start;
    return t;
}

// Cross-feature index generation for a whole launch (Section 3.3, "real-time generation" from the candidate's
// attribute): xb[pos][f] = bucket of candidate pos in field f, or kNoBucket for an id outside the item table.  Done
// once per call so that the layer kernel's gather threads only look the bucket up.  Ids in mapped host memory are copied
// to ids_copy on the way, for the kernels that follow; candidates that are grouped by category are placed on the way (pl.where:
// pos becomes the grouped position; F = 0 does nothing else).
// POW2: the number of buckets is a power of two (a mask, with nothing of the other form's multiplications beside it).
constexpr uint32_t kNoBucket = 0xFFFFu;
template <bool POW2>
__global__ void __launch_bounds__(256) k_cross_buckets(const int32_t *__restrict__ ids, int64_t total, int64_t M, int F, int B,
                                                        uint64_t b_inv, int mode, uint16_t *__restrict__ xb, int32_t *__restrict__ ids_copy, const SimPlace pl, int late)
{
    if (!late) grid_dep_wait();
    grid_dep_launch();
    // A warp takes 32 consecutive candidates: one coalesced read of their ids (128 bytes, also the right size for a read
    // across the bus), then 32 F hashes that depend on nothing else, two per thread and round, leaving as one 4-byte store
    // per thread (an odd number of fields, possible only with embeddings of 64 columns and more, takes one hash per round).
    const int lane = threadIdx.x & 31, step = F & 1 ? 1 : 2;
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < total; base += n_warps * 32) {
        int my = -1, to = lane;   // to: the candidate's row of xb, counted from base
        if (base + lane < total) {
            my = ids[base + lane];
            if (ids_copy && blockIdx.y == 0) ids_copy[base + lane] = my;
            if (pl.where) {
                const int2 w = pl.where[base + lane];
                const int at = pl.grp_start[w.x] + w.y;
                to = at - (int)base;
                if (blockIdx.y == 0) pl.ids[at] = my, pl.out_index[at] = (int)base + lane;
            }
        }
        const int n = (int)min((int64_t)32, total - base) * F;
        uint16_t *out = xb + base * F;
        // small launches spread a warp's hashes over gridDim.y warps (the ids are then read that many times)
        for (int i0 = 32 * step * (int)blockIdx.y; i0 < 32 * F; i0 += 32 * step * (int)gridDim.y) {
            const int i = i0 + lane * step, c = i / F, f = i - c * F;
            const int id = __shfl_sync(0xffffffffu, my, c & 31), row = __shfl_sync(0xffffffffu, to, c & 31);
            const bool good = id >= 0 && (int64_t)id < M;
            uint32_t bk[2] = {kNoBucket, kNoBucket};
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (good && q < step) {
                    if (mode == AIF_BUCKET_MOD) bk[q] = (uint32_t)(id % B);
                    else {
                        const uint64_t h = mix64((uint64_t)id, (uint64_t)(f + q));
                        if (POW2) bk[q] = (uint32_t)h & (uint32_t)(B - 1);
                        else {
                            // Barrett reduction with b_inv = floor(2^64 / B): the estimated quotient is the true one or one less, as
                            // h (2^64 / B - b_inv) / 2^64 < 1.  With a 64-bit remainder each, 2 x 10^7 hashes took 130 us, so 62.
                            const uint32_t r = (uint32_t)h - (uint32_t)__umul64hi(h, b_inv) * (uint32_t)B;   // below 2 B: 32 bits are enough
                            bk[q] = r >= (uint32_t)B ? r - (uint32_t)B : r;
                        }
                    }
                }
            if (i >= n) continue;
            uint16_t *o = out + (int64_t)row * F + f;
            if (step == 2) *reinterpret_cast<uint32_t *>(o) = bk[0] | (bk[1] << 16);
            else *o = (uint16_t)bk[0];
        }
    }
    if (late && (blockIdx.x | blockIdx.y) == 0) grid_dep_wait();
}

// Tile table of a launch over several requests: one thread per tile does the search of the request table that every
// role of every kernel would otherwise repeat per tile (a chain of dependent loads on the critical path of the MMA
// issuers).
__global__ void __launch_bounds__(256) k_tile_table(ScoreLaunch sl, int mini_batch, TileDev *__restrict__ out)
{
    grid_dep_launch();
    grid_dep_wait();
    const int tile = blockIdx.x * blockDim.x + threadIdx.x;
    if (tile >= sl.n_tiles) return;
    out[tile] = tile_entry(sl, tile, mini_batch);
}

// Rows of a chunk of the first layer's input, brought into a stage by one warp.  Lane l: 16-byte slot l % 8 of the 128-byte rows
// l / 8 + 4 i.  The sources of a chunk are one number per row, the item id or the bucket(s) of the chunk's field(s): lane l
// fetches those of rows l + 32 j with coalesced loads (fetch), the copying lanes get them by shuffle (copy).
struct ChunkRows {
    int kind;
    int32_t v[4];           // per row lane + 32 j: id as read, or bucket (both fields' buckets); -1: zero row
    const uint8_t *bp;      // this lane's 16 bytes of row 0 of the table the rows come from
    const uint16_t *xb;     // narrow fields: this lane's field of the tile's first row of buckets
    uint32_t row_bytes;     // of that table
    int cnt;                // rows of the tile
    int tma_x, tma_y;       // dense chunk; tma_x < 0: the tile does not exist
};
struct RowGather {
    int lane, sub, r0;
    uint32_t swz0, swz1;   // row & 7 alternates between r0 and r0 + 4
    bool two;          // two fields per chunk; wider embeddings: one field spans one or more chunks
    bool narrow;       // four and more fields per chunk: the copying lanes look their buckets up themselves
    __device__ __forceinline__ RowGather(const LayerParams &p, int l)
        : lane(l), sub(l & 7), r0(l >> 3), swz0((uint32_t)((sub ^ r0) << 4)), swz1((uint32_t)((sub ^ (r0 + 4)) << 4)), two(p.dc == 32), narrow(p.dc < 32)
    {
    }
    __device__ __forceinline__ void fetch(ChunkRows &c, const LayerParams &p, int kc, const TileInfo &t) const
    {
        const ChunkSrc src = p.src[kc];
        c.kind = src.kind, c.cnt = t.cnt;
        if (src.kind == SRC_DENSE) {
            // rows beyond the tile bring other candidates' values along; their results are never stored
            c.tma_x = t.cnt > 0 ? src.off >> 1 : -1, c.tma_y = (int)t.pos0;
        } else if (src.kind == SRC_ITEM) {
            c.bp = p.E + src.off + sub * 16, c.row_bytes = (uint32_t)p.e_row_bytes;
#pragma unroll
            for (int j = 0; j < 4; ++j) c.v[j] = lane + 32 * j < t.cnt ? p.sl.ids[t.pos0 + lane + 32 * j] : -1;
        } else if (narrow) {
            const int col = src.off + sub * 8, f = col / p.dc;
            c.row_bytes = (uint32_t)p.dc * 2;
            c.bp = p.T0 + (size_t)t.rq.slot * p.slot_bytes + ((size_t)f * p.B * p.dc + (col - f * p.dc)) * 2;
            c.xb = p.xb + (size_t)t.pos0 * p.F + f;
        } else {
            const int f = src.off / p.dc, col = two ? (sub & 3) * 8 : src.off - f * p.dc + sub * 8;
            c.row_bytes = (uint32_t)p.dc * 2;
            c.bp = p.T0 + (size_t)t.rq.slot * p.slot_bytes + ((size_t)(f + (two ? sub >> 2 : 0)) * p.B * p.dc + col) * 2;
            const uint16_t *xb = p.xb + (size_t)t.pos0 * p.F + f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                c.v[j] = -1;
                if (lane + 32 * j < t.cnt) {
                    const uint16_t *w = xb + (size_t)(lane + 32 * j) * p.F;
                    // F is even where dc = 32; a bucket that does not exist is 0xFFFF, both of a pair at once
                    c.v[j] = two ? __ldg(reinterpret_cast<const int32_t *>(w)) : (int32_t)((uint32_t)__ldg(w) | 0xFFFF0000u);
                }
            }
        }
    }
    // a gathered chunk (not SRC_DENSE); c is used up
    __device__ __forceinline__ void copy(ChunkRows &c, const LayerParams &p, uint32_t dst0, bool first) const
    {
        // row r0 + 4 i: register i / 8 of lane r0 + 4 (i % 8)
        if (c.kind == SRC_ITEM) {
            bool bad = false;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c.v[j] < 0 || (int64_t)c.v[j] >= p.M) {
                    bad |= lane + 32 * j < c.cnt;
                    c.v[j] = -1;
                }
            if (bad && p.check_ids && first) atomicOr(p.sl.status, AIF_STATUS_BAD_ID);
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const int v = __shfl_sync(0xffffffffu, c.v[i >> 3], r0 + 4 * (i & 7));
                cp_async16(dst0 + (uint32_t)(i * 512) + (i & 1 ? swz1 : swz0), c.bp + (size_t)(uint32_t)max(v, 0) * c.row_bytes, v >= 0 ? 16u : 0u);
            }
        } else if (narrow) {
#pragma unroll 1
            for (int i0 = 0; i0 < 32; i0 += 8) {
                uint32_t v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int row = r0 + 4 * (i0 + i);
                    v[i] = row < c.cnt ? (uint32_t)__ldg(c.xb + (size_t)row * p.F) : kNoBucket;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const bool on = v[i] != kNoBucket;
                    cp_async16(dst0 + (uint32_t)((i0 + i) * 512) + (i & 1 ? swz1 : swz0), c.bp + (size_t)(on ? v[i] : 0u) * c.row_bytes, on ? 16u : 0u);
                }
            }
        } else {
            const uint32_t pick = two && sub >= 4 ? 0x4432u : 0x4410u;   // byte permute: the pair's upper or lower half
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const uint32_t v = __byte_perm((uint32_t)__shfl_sync(0xffffffffu, c.v[i >> 3], r0 + 4 * (i & 7)), 0u, pick);
                const bool on = v != kNoBucket;
                cp_async16(dst0 + (uint32_t)(i * 512) + (i & 1 ? swz1 : swz0), c.bp + (size_t)(on ? v : 0u) * c.row_bytes, on ? 16u : 0u);
            }
        }
    }
};

// ---- the layer kernel ---------------------------------------------------------------------------------------------
// Every product spans two SMs (cta_group::2).  What bounds a layer is the rate at which an SM takes in operands (59 bytes per
// clock).  With both tiles of an item in one SM, which that rate asks for, their accumulators filled tensor memory and the
// epilogue was exposed, 6 k of 22 k cycles per item (64 requests of 10^4 candidates, first layer).  Here a CTA holds its tile's
// rows and half of the weight slice, 32 KB per 64-column chunk for 512 cycles of products, the same intake per flop, and one
// 256-column accumulator: two fit, and the epilogue of an item runs under the products of the next.
// First layer of 64 x 10^4 candidates (K = 768, 512 outputs): 471 -> 386 us; of 256 x 4000 candidates at d = 256 (K = 2560,
// 1024 outputs): 5.17 -> 4.11 ms; second layers 176 -> 140 and 1125 -> 800 us.
// Slices narrower than 256 are rounded up to a multiple of 64 (each CTA brings half of the weight rows, its epilogue warps
// take whole 32-column pieces); weight rows beyond the last output arrive as zeros.
// Roles per CTA (512 threads): 8 epilogue warps (two per quarter of the rows, half of the columns each), the MMA warp (the
// even CTA's lane issues), 6 gather warps and one weight warp.  One ring of six stages, rows and weights of a chunk together,
// and one arrival per CTA that both have landed: the issuing lane has one wait per chunk, which is shorter than the product it
// leaves in the queue.
struct PairCfg {
    static constexpr int kStages = 6, kStage = 2 * kABytes;
    // one gather warp per stage: a warp meets every phase of its own stage in turn, so that a wait on the phase's parity can
    // never be answered by an older phase
    static constexpr int kEpiWarps = 8, kMmaWarp = 8, kProdWarp0 = 9, kProdWarps = kStages, kBWarp = kProdWarp0 + kProdWarps;
    static constexpr int kThreads = (kBWarp + 1) * 32;
    static constexpr int kOffSlab = kStages * kStage, kOffMisc = kOffSlab + kEpiWarps * 2048;
    // barriers and the tensor-memory slot | bias, output weights [256] | dot products of the upper halves [128]
    static constexpr size_t kSmem = 1024 + kOffMisc + 256 + 2 * 256 * 4 + 128 * 4;
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

__global__ void __launch_bounds__(PairCfg::kThreads, 1) k_layer_pair(const __grid_constant__ CUtensorMap tmapB,
                                                                     const __grid_constant__ CUtensorMap tmapOut,
                                                                     const __grid_constant__ CUtensorMap tmapA, const LayerParams p)
{
    using C = PairCfg;
    constexpr int kS = C::kStages;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    unsigned char *out_stage = base + C::kOffSlab;
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + C::kOffMisc);
    uint64_t *full = bars, *empty = full + kS, *landed = empty + kS, *acc_full = landed + kS, *acc_empty = acc_full + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 2);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    float *bias_s = reinterpret_cast<float *>(base + C::kOffMisc + 256), *wout_s = bias_s + 256, *dot_s = wout_s + 256;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank();   // 0: issues the products

    if (tid == 0) {
        for (int s = 0; s < kS; ++s) {
            mbar_init(smem_u32(full + s), 2);      // a gather warp of each CTA (used in the even one)
            mbar_init(smem_u32(landed + s), 2);    // TMA copies of this CTA: announced by the weight lane and by the gather warp
            mbar_init(smem_u32(empty + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(acc_full + b), 1);
            mbar_init(smem_u32(acc_empty + b), 2 * C::kEpiWarps);   // the epilogue warps of both CTAs (used in the even one)
        }
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == C::kMmaWarp) tmem_alloc_pair(smem_u32(tmem_slot), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // the other CTA's barriers exist
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    grid_dep_launch();
    if (warp != C::kBWarp && !p.sl.late) grid_dep_wait();   // the weights are older than any launch this one may overlap
    const int n_tiles = p.sl.n_tiles;
    const int n_items = ((n_tiles + 1) / 2) * p.n_nchunks;
    const int item0 = (int)(blockIdx.x >> 1), item_step = (int)(gridDim.x >> 1);

    if (warp < C::kEpiWarps) {
        // ===================== epilogue =====================
        const int wq = warp & 3, half = warp >> 2;
        const int row = wq * 32 + lane;              // TMEM lane = candidate row of the tile
        const int hc = p.n_cols >> 1, col_lo = half * hc;
        unsigned char *sb = out_stage + warp * 2048;   // staging slab of 32 rows x 64 bytes, 64-byte swizzle (the layout tmapOut expects)
        const int l4 = lane & 3, r8 = lane >> 2, wrow0 = wq * 32;
        uint32_t empty_addr[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) empty_addr[b] = cluster_addr(smem_u32(acc_empty + b), 0u);
        // a wait that ran out in an earlier kernel of this call left its outputs unwritten: logits computed from them are
        // replaced by NaN
        const bool poisoned = p.epi == EPI_DOT && (*reinterpret_cast<volatile const uint32_t *>(p.sl.status) & AIF_STATUS_TIMEOUT) != 0u;
        int it = 0;
        for (int item = item0; item < n_items; item += item_step, ++it) {
            const int grp = item / p.n_nchunks, n0 = (item - grp * p.n_nchunks) * p.n_cols;
            const int buf = it & 1;
            const TileInfo t = decode_tile(p, grp * 2 + rank, n_tiles);
            const bool valid = row < t.cnt;
            int id = -1;
            if (p.epi == EPI_DOT && half == 0 && valid) id = p.sl.ids[t.pos0 + row];
            if (t.cnt > 0) {
                const float *bias = p.bias_from_slot ? p.sl.slots[t.rq.slot].p_u : p.bias;
                if (tid < p.n_cols) {
                    const bool is_out = n0 + tid < p.n_out;
                    bias_s[tid] = is_out ? bias[n0 + tid] : 0.f;
                    if (p.epi == EPI_DOT) wout_s[tid] = is_out ? __bfloat162float(p.w_out[n0 + tid]) : 0.f;
                }
            }
            named_bar_sync(1, 256);
            // a wait that ran out is carried to the barrier at the end of the item, so that the warps leave together
            const bool got = __all_sync(0xffffffffu, mbar_wait(smem_u32(acc_full + buf), (uint32_t)((it >> 1) & 1), abort_flag));
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)wrow0 << 16) + (uint32_t)(buf * 256 + col_lo);
            float dot = 0.f;
            if (got && t.cnt > 0 && p.epi == EPI_STORE) {
                // The accumulator is read in the 16x256b shape: a thread owns two columns (per group of eight) over four rows
                // and needs eight bias values per 32 columns.  Three instructions per pair of outputs: bias added to both
                // (f32x2), rounded to bf16, ReLU on the rounded pair (rounding is monotonic and keeps zero).
                const __nv_bfloat162 floor2 = __float2bfloat162_rn(p.linear_out ? -INFINITY : 0.f);
                for (int c0 = 0; c0 < hc && n0 + col_lo + c0 < p.n_out; c0 += 32) {   // stored widths are multiples of 32
                    uint32_t ra[16], rb[16];
                    tmem_ld16x256(taddr + (uint32_t)c0, ra);                    // rows 0..15 of this warp's 32
                    tmem_ld16x256(taddr + (16u << 16) + (uint32_t)c0, rb);      // rows 16..31
                    uint64_t bias2[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) bias2[j] = *reinterpret_cast<const uint64_t *>(bias_s + col_lo + c0 + 8 * j + 2 * l4);
                    if (lane == 0) bulk_wait_read<0>();   // the store that last read the slab is done with it
                    tmem_ld_wait();
                    __syncwarp();
                    auto emit = [&](const uint32_t (&r)[16], int row_h) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                float x0, x1;
                                unpack_f32x2(add_f32x2(pack_f32x2(__uint_as_float(r[4 * j + 2 * q]), __uint_as_float(r[4 * j + 2 * q + 1])), bias2[j]), x0, x1);
                                const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(x0, x1), floor2);
                                const int rr = row_h + r8 + 8 * q;
                                *reinterpret_cast<uint32_t *>(sb + rr * 64 + ((j ^ ((rr >> 1) & 3)) << 4) + 4 * l4) = *reinterpret_cast<const uint32_t *>(&h);
                            }
                    };
                    emit(ra, 0);
                    emit(rb, 16);
                    if (wrow0 + 32 <= t.cnt) {
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(&tmapOut, smem_u32(sb), n0 + col_lo + c0, (int)(t.pos0 + wrow0));
                            bulk_commit();
                        }
                    } else {   // ragged last tile of a request or mini-batch: guarded stores
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int rr = 8 * j + (lane >> 2), q = lane & 3;
                            const uint4 v = *reinterpret_cast<const uint4 *>(sb + rr * 64 + ((q ^ ((rr >> 1) & 3)) << 4));
                            if (wrow0 + rr < t.cnt)
                                *reinterpret_cast<uint4 *>(p.out + (size_t)(t.pos0 + wrow0 + rr) * p.out_stride + n0 + col_lo + c0 + q * 8) = v;
                        }
                        __syncwarp();
                    }
                }
            } else if (got && t.cnt > 0 && p.epi == EPI_DOT) {
                // Last hidden layer: ReLU(x + b) . w_out per row over this warp's columns, in the same shape; the four threads
                // of a row are joined by shuffles, the two halves of the columns through shared memory.
                uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};   // rows r8 + 8 i, two columns each
                for (int c0 = 0; c0 < hc; c0 += 32) {
                    uint32_t ra[16], rb[16];
                    tmem_ld16x256(taddr + (uint32_t)c0, ra);
                    tmem_ld16x256(taddr + (16u << 16) + (uint32_t)c0, rb);
                    uint64_t bias2[4], w2[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int col = col_lo + c0 + 8 * j + 2 * l4;
                        bias2[j] = *reinterpret_cast<const uint64_t *>(bias_s + col);
                        w2[j] = *reinterpret_cast<const uint64_t *>(wout_s + col);
                    }
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            float x0, x1, y0, y1;
                            unpack_f32x2(add_f32x2(pack_f32x2(__uint_as_float(ra[4 * j + 2 * q]), __uint_as_float(ra[4 * j + 2 * q + 1])), bias2[j]), x0, x1);
                            unpack_f32x2(add_f32x2(pack_f32x2(__uint_as_float(rb[4 * j + 2 * q]), __uint_as_float(rb[4 * j + 2 * q + 1])), bias2[j]), y0, y1);
                            acc[q] = fma_f32x2(pack_f32x2(fmaxf(x0, 0.f), fmaxf(x1, 0.f)), w2[j], acc[q]);
                            acc[2 + q] = fma_f32x2(pack_f32x2(fmaxf(y0, 0.f), fmaxf(y1, 0.f)), w2[j], acc[2 + q]);
                        }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float lo, hi;
                    unpack_f32x2(acc[i], lo, hi);
                    float v = lo + hi;
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    // row 8 i + r8 of this warp's 32 belongs to lane 8 i + r8; lane 4 r8 (among others) holds its sum
                    v = __shfl_sync(0xffffffffu, v, 4 * (lane & 7));
                    if ((lane >> 3) == i) dot = v;
                }
                if (half == 1) dot_s[row] = dot;
            } else if (got && t.cnt > 0) {   // EPI_SIGN
                for (int c0 = 0; c0 < hc && n0 + col_lo + c0 < p.n_out; c0 += 32) {
                    uint32_t r[32];
                    tmem_ld32(taddr + (uint32_t)c0, r);
                    tmem_ld_wait();
                    // eq. 5: one bit per output, set where the projection is positive; eight bits per byte, first bit most
                    // significant
                    uint32_t word = 0u;
#pragma unroll
                    for (int i = 0; i < 32; ++i) word |= (__uint_as_float(r[i]) > 0.f ? 1u : 0u) << (8 * (i >> 3) + 7 - (i & 7));
                    if (valid) *reinterpret_cast<uint32_t *>(p.sig_out + (size_t)(t.pos0 + row) * (p.out_stride >> 3) + ((n0 + col_lo + c0) >> 3)) = word;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (got && lane == 0) mbar_arrive_cluster(empty_addr[buf]);
            const bool out = named_bar_or(1, 256, !got);   // also orders dot_s
            if (p.epi == EPI_DOT && half == 0 && valid) {
                float logit = dot + dot_s[row] + p.b_out[0];
                if (p.emit_sigmoid) logit = 1.0f / (1.0f + expf(-logit));
                // no number for an id outside the table, nor for a tile whose inputs never arrived (here or in an earlier
                // kernel of the call: the status word says so)
                if (id < 0 || (int64_t)id >= p.M || out || poisoned) logit = __int_as_float(0x7fc00000);
                p.sl.logits[p.sl.out_index ? (int64_t)p.sl.out_index[t.pos0 + row] : t.pos0 + row] = logit;
            }
            if (out) break;
        }
        if (lane == 0) bulk_wait<0>();   // all tile stores of this warp have reached global memory
    } else if (warp == C::kMmaWarp) {
        if (lane == 0 && rank == 0) {
            // ===================== MMA issuer =====================
            const uint32_t idesc = umma_idesc_bf16(2 * kTcTile, p.n_cols);
            const uint64_t adesc0 = umma_desc_sw128(smem_u32(base)), bdesc0 = umma_desc_sw128(smem_u32(base + kABytes));
            int it = 0, s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int item = item0; ok && item < n_items; item += item_step, ++it) {
                const int buf = it & 1;
                // the accumulator must have been drained by both CTAs' epilogues of its previous use
                if (!mbar_wait(smem_u32(acc_empty + buf), (uint32_t)((it >> 1) & 1) ^ 1u, abort_flag)) break;
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256);
                for (int kc = 0; kc < p.n_k; ++kc) {
                    if (!mbar_wait(smem_u32(full + s), ph, abort_flag)) {
                        ok = false;
                        break;
                    }
                    fence_proxy_async();   // gathered rows were written by cp.async (generic proxy)
                    tc_fence_after();
                    const uint64_t off = (uint64_t)(uint32_t)(s * (C::kStage >> 4));
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)   // 4 x K=16 inside the 64-column chunk: +32 bytes (2 units) per step
                        umma_bf16_pair(d_tmem, adesc0 + off + 2 * kk, bdesc0 + off + 2 * kk, idesc, (kc | kk) != 0 ? 1u : 0u);
                    umma_commit_pair(smem_u32(empty + s));
                    if (kc == p.n_k - 1) umma_commit_pair(smem_u32(acc_full + buf));
                    if (++s == kS) s = 0, ph ^= 1u;
                }
            }
        }
        __syncwarp();
    } else if (warp < C::kBWarp) {
        // ===================== A producers: every warp fills the stage of its number, all 128 rows of a chunk =====================
        // Lane l: 16-byte slot l % 8 of the 128-byte rows l / 8 + 4 i.  The sources of a chunk are one number per row, the item
        // id or the bucket(s) of the chunk's field(s): lane l fetches those of rows l + 32 j with coalesced loads while the
        // previous chunk of this warp is landing, the copying lanes get them by shuffle.  What the fetch itself needs, the
        // tile's place, is requested one chunk earlier still: a fetch that had to wait for it took 1250 to 3000 of a chunk's
        // 3300 cycles.  A warp waits for its own copies (five others have theirs in flight meanwhile) and tells the issuer
        // with one arrival: an arrival per gathering thread (256 serial operations on the stage's barrier) cost more than the
        // 512 cycles of products a chunk is.
        const RowGather g(p, lane);
        const int n_k = p.n_k;
        const int s = warp - C::kProdWarp0;
        const uint32_t dst0 = smem_u32(base + s * C::kStage) + (uint32_t)(g.r0 * 128);
        struct Place {
            int item, kc;
        };
        auto step = [&](Place &q, int by) {
            q.kc += by;
            while (q.kc >= n_k) q.kc -= n_k, q.item += item_step;
        };
        auto tile_of = [&](const Place &q) { return decode_tile(p, q.item < n_items ? (q.item / p.n_nchunks) * 2 + rank : n_tiles, n_tiles); };
        uint32_t ph = 0;
        Place cur{item0, 0}, nxt;
        step(cur, s);
        nxt = cur, step(nxt, C::kProdWarps);
        ChunkRows c;
        if (cur.item < n_items) g.fetch(c, p, cur.kc, tile_of(cur));
        TileInfo tn = tile_of(nxt);
        while (cur.item < n_items) {
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(empty + s), ph ^ 1u, abort_flag))) break;
            const bool gathered = c.kind != SRC_DENSE;
            if (!gathered) {
                if (lane == 0) {
                    if (c.tma_x >= 0) {
                        mbar_expect_tx(smem_u32(landed + s), (uint32_t)kABytes);
                        tma_load_2d(smem_u32(base + s * C::kStage), &tmapA, smem_u32(landed + s), c.tma_x, c.tma_y);
                    } else
                        mbar_arrive(smem_u32(landed + s));
                }
            } else {
                if (lane == 0) mbar_arrive(smem_u32(landed + s));
                g.copy(c, p, dst0, cur.kc == 0);
                cp_async_commit();
            }
            cur = nxt;
            step(nxt, C::kProdWarps);
            if (cur.item < n_items) g.fetch(c, p, cur.kc, tn);   // these loads are in flight while the copies land
            tn = tile_of(nxt);
            if (gathered) {
                cp_async_wait<0>();
                fence_proxy_async();   // written by cp.async (generic proxy), read by the products through the async proxy
            }
            __syncwarp();
            bool ok = true;
            if (lane == 0) {
                ok = mbar_wait(smem_u32(landed + s), ph, abort_flag);   // the stage's weights, and a dense chunk's rows
                if (ok) mbar_arrive_cluster(cluster_addr(smem_u32(full + s), 0u));
            }
            if (!__all_sync(0xffffffffu, ok)) break;
            ph ^= 1u;
        }
        cp_async_wait_all();
    } else {
        // ===================== B producer (TMA): this CTA's half of the slice's weight rows =====================
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            const int rows = p.n_cols >> 1;
            for (int item = item0; ok && item < n_items; item += item_step) {
                const int n0 = (item % p.n_nchunks) * p.n_cols + rank * rows;
                for (int kc = 0; kc < p.n_k; ++kc) {
                    if (!mbar_wait(smem_u32(empty + s), ph ^ 1u, abort_flag)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(smem_u32(landed + s), (uint32_t)rows * 128u);
                    tma_load_2d(smem_u32(base + s * C::kStage + kABytes), &tmapB, smem_u32(landed + s), kc * 64, n0);
                    if (++s == kS) s = 0, ph ^= 1u;
                }
            }
        }
        __syncwarp();
    }

    // ---- teardown: everybody arrives here, also after an abort; neither CTA leaves while the other may still reach it
    if (*abort_flag) {
        if (tid == 0) atomicOr(p.sl.status, AIF_STATUS_TIMEOUT);
        // let copies and MMAs that are still in flight land before shared memory and TMEM go away
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == C::kMmaWarp) tmem_dealloc_pair(tmem_base, 512);
    if (p.sl.late && blockIdx.x == 0) grid_dep_wait();
}

// ---- both layers of a two-layer MLP -------------------------------------------------------------------------------
// Launches of at most one tile per SM, 512 and at most 256 units: the whole MLP of a tile in one kernel.  In the layer kernel
// 10^4 candidates are 80 items of the first layer on 74 pairs of SMs, two rounds for little more than one, and either
// layer's start and end (tile look-up, first rows, last accumulators, stores) is as long as its products.  Here a CTA keeps its tile:
// both 256-column accumulators of the first layer fill its tensor memory, the activations go back there as bf16 (A operand of
// the second layer) over accumulator columns already read, and nothing but the logits is written.  Products span a pair of CTAs
// as in the layer kernel (the two tiles may belong to different requests): with whole weight slices per CTA, operand intake
// (1360 cycles per 64-column chunk at 59 bytes per clock) would bound it, not the products (1024).
// Roles per CTA (448 threads): 8 epilogue warps (group g: output slice g, later half g of the second layer's units), the MMA warp,
// 4 gather warps, one per stage, one weight warp.  A stage is a 64-column chunk of the rows and of both slices' weights, later
// two chunks of the second layer's weights.  The first layer's accumulators start from the bias instead of zero.
// Tensor memory: accumulators [0, 256) and [256, 512), packed activations [0, 128) and [384, 512), second layer [128, 128 + H2).
struct MlpCfg {
    static constexpr int kH1 = 512;
    static constexpr int kStages = 4, kStage = 3 * kABytes;
    static constexpr int kMmaWarp = 8, kProdWarp0 = 9, kBWarp = kProdWarp0 + kStages, kThreads = (kBWarp + 1) * 32;
    static constexpr int kOffMisc = kStages * kStage;
    // barriers and the tensor-memory slot | bias, output weights [256] | dot products of the upper halves [128]
    static constexpr size_t kSmem = 1024 + kOffMisc + 256 + (2 * 256 + 128) * 4;
    static_assert(kSmem <= 227 * 1024, "shared memory");
};
struct MlpParams {
    LayerParams l;   // the first layer's
    int32_t H2;
    const float *b2;
};

__global__ void __launch_bounds__(MlpCfg::kThreads, 1) k_mlp_pair(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapW1,
                                                                  const __grid_constant__ CUtensorMap tmapW2, const __grid_constant__ MlpParams mp)
{
    using C = MlpCfg;
    constexpr int kS = C::kStages;
    const LayerParams &p = mp.l;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + C::kOffMisc);
    uint64_t *full = bars, *empty = full + kS, *landed = empty + kS, *preset = landed + kS, *acc1 = preset + 1, *h1 = acc1 + 1, *acc2 = h1 + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc2 + 1);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    float *bias_s = reinterpret_cast<float *>(base + C::kOffMisc + 256), *wout_s = bias_s + 256, *dot_s = wout_s + 256;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank();   // 0: issues the products

    if (tid == 0) {
        for (int s = 0; s < kS; ++s) {
            mbar_init(smem_u32(full + s), 2);      // a gather warp of each CTA (used in the even one)
            mbar_init(smem_u32(landed + s), 2);    // TMA copies of this CTA: announced by the weight lane and by the gather warp
            mbar_init(smem_u32(empty + s), 1);
        }
        mbar_init(smem_u32(preset), 16);           // the epilogue warps of both CTAs (used in the even one)
        mbar_init(smem_u32(h1), 16);
        mbar_init(smem_u32(acc1), 1);
        mbar_init(smem_u32(acc2), 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == C::kMmaWarp) tmem_alloc_pair(smem_u32(tmem_slot), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // the other CTA's barriers exist
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    grid_dep_launch();
    const int n_stages = p.n_k + C::kH1 / 128;   // uses of the ring
    if (warp != C::kBWarp) grid_dep_wait();      // the weights are older than any launch this one may overlap

    if (warp < 8) {
        // ===================== epilogues: one thread per row in each group =====================
        const int g = warp >> 2, wq = warp & 3, row = wq * 32 + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
        bool ok = true;
        auto wait = [&](uint64_t *b) {
            const bool got = mbar_wait(smem_u32(b), 0u, abort_flag);
            ok = __all_sync(0xffffffffu, ok && got);
        };
        auto arrive_even = [&](uint64_t *b) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_addr(smem_u32(b), 0u));
        };
        const TileInfo t = decode_tile(p, (int)blockIdx.x, p.sl.n_tiles);
        {
            const float4 *pu = reinterpret_cast<const float4 *>(p.sl.slots[t.rq.slot].p_u + 256 * g);
#pragma unroll 1
            for (int c = 0; c < 256; c += 32) {
                uint32_t r[32];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 v = pu[c / 4 + j];
                    r[4 * j] = __float_as_uint(v.x), r[4 * j + 1] = __float_as_uint(v.y), r[4 * j + 2] = __float_as_uint(v.z), r[4 * j + 3] = __float_as_uint(v.w);
                }
                tmem_st32(lane_base + (uint32_t)(256 * g + c), r);
            }
            tmem_st_wait();
            arrive_even(preset);
        }
        // a wait that ran out in an earlier kernel of this call left its outputs unwritten: logits computed from them are
        // replaced by NaN
        const bool poisoned = (*reinterpret_cast<volatile const uint32_t *>(p.sl.status) & AIF_STATUS_TIMEOUT) != 0u;
        const bool valid = row < t.cnt;
        int id = -1;
        if (g == 0 && valid) id = p.sl.ids[t.pos0 + row];
        if (tid < mp.H2) bias_s[tid] = mp.b2[tid], wout_s[tid] = __bfloat162float(p.w_out[tid]);
        named_bar_sync(1, 256);
        // ---- first layer: slice g, ReLU, 32 accumulator columns -> 16 columns of packed bf16, over accumulator columns already
        // read (slice 0 upwards, slice 1 downwards: the 256 columns in between become free)
        wait(acc1);
        tc_fence_after();
        if (ok) {
            uint32_t ra[32], rb[32];
            const uint32_t col0 = lane_base + (uint32_t)(g * 256);
            auto finish = [&](const uint32_t (&r)[32], int c) {
                uint32_t packed[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(__uint_as_float(r[2 * q]), __uint_as_float(r[2 * q + 1])), __float2bfloat162_rn(0.f));
                    packed[q] = *reinterpret_cast<const uint32_t *>(&h);
                }
                tmem_st16(lane_base + (uint32_t)((g ? 384 : 0) + 16 * c), packed);
            };
            auto chunk_of = [&](int i) { return g ? 7 - i : i; };
            tmem_ld32(col0 + (uint32_t)(32 * chunk_of(0)), ra);
#pragma unroll 1
            for (int i = 0; i < 8; i += 2) {
                tmem_ld_wait();
                tmem_ld32(col0 + (uint32_t)(32 * chunk_of(i + 1)), rb);
                finish(ra, chunk_of(i));
                tmem_ld_wait();
                if (i + 2 < 8) tmem_ld32(col0 + (uint32_t)(32 * chunk_of(i + 2)), ra);
                finish(rb, chunk_of(i + 1));
            }
            tmem_st_wait();
        }
        arrive_even(h1);
        // ---- second layer: half g of the units, bias, ReLU, reduced against w_out
        wait(acc2);
        tc_fence_after();
        float dot = 0.f;
        if (ok) {
            const int hn = mp.H2 >> 1;   // a multiple of 32
            const uint32_t col0 = lane_base + 128u + (uint32_t)(g * hn);
            float d4[4] = {0.f, 0.f, 0.f, 0.f};
            uint32_t ra[32], rb[32];
            auto reduce = [&](const uint32_t (&r)[32], int c0) {
                const float4 *b4 = reinterpret_cast<const float4 *>(bias_s + g * hn + c0), *w4 = reinterpret_cast<const float4 *>(wout_s + g * hn + c0);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float4 b = b4[q], w = w4[q];
                    d4[0] = fmaf(fmaxf(__uint_as_float(r[4 * q]) + b.x, 0.f), w.x, d4[0]);
                    d4[1] = fmaf(fmaxf(__uint_as_float(r[4 * q + 1]) + b.y, 0.f), w.y, d4[1]);
                    d4[2] = fmaf(fmaxf(__uint_as_float(r[4 * q + 2]) + b.z, 0.f), w.z, d4[2]);
                    d4[3] = fmaf(fmaxf(__uint_as_float(r[4 * q + 3]) + b.w, 0.f), w.w, d4[3]);
                }
            };
            tmem_ld32(col0, ra);
#pragma unroll 1
            for (int c0 = 0; c0 < hn; c0 += 64) {
                tmem_ld_wait();
                if (c0 + 32 < hn) tmem_ld32(col0 + (uint32_t)(c0 + 32), rb);
                reduce(ra, c0);
                if (c0 + 32 < hn) {
                    tmem_ld_wait();
                    if (c0 + 64 < hn) tmem_ld32(col0 + (uint32_t)(c0 + 64), ra);
                    reduce(rb, c0 + 32);
                }
            }
            dot = (d4[0] + d4[1]) + (d4[2] + d4[3]);
        }
        if (g == 1) dot_s[row] = dot;
        const bool out = named_bar_or(1, 256, !ok);   // also orders dot_s
        if (g == 0 && valid) {
            float logit = dot + dot_s[row] + p.b_out[0];
            if (p.emit_sigmoid) logit = 1.0f / (1.0f + expf(-logit));
            // no number for an id outside the table, nor for a tile whose inputs never arrived (here or in an earlier kernel of
            // the call: the status word says so)
            if (id < 0 || (int64_t)id >= p.M || out || poisoned) logit = __int_as_float(0x7fc00000);
            p.sl.logits[p.sl.out_index ? (int64_t)p.sl.out_index[t.pos0 + row] : t.pos0 + row] = logit;
        }
    } else if (warp == C::kMmaWarp) {
        if (lane == 0 && rank == 0) {
            // ===================== MMA issuer =====================
            constexpr uint32_t idesc1 = umma_idesc_bf16(2 * kTcTile, 256);
            const uint32_t idesc2 = umma_idesc_bf16(2 * kTcTile, mp.H2);
            const uint64_t desc0 = umma_desc_sw128(smem_u32(base));
            bool ok = mbar_wait(smem_u32(preset), 0u, abort_flag);
#pragma unroll 1
            for (int i = 0; ok && i < n_stages; ++i) {
                const int s = i % kS;
                if (i == p.n_k) {
                    umma_commit_pair(smem_u32(acc1));
                    if (!mbar_wait(smem_u32(h1), 0u, abort_flag)) ok = false;
                }
                if (!ok || !mbar_wait(smem_u32(full + s), (uint32_t)((i / kS) & 1), abort_flag)) {
                    ok = false;
                    break;
                }
                fence_proxy_async();   // gathered rows were written by cp.async (generic proxy)
                tc_fence_after();
                const uint64_t d = desc0 + (uint64_t)(uint32_t)(s * (C::kStage >> 4));
                if (i < p.n_k) {
#pragma unroll
                    for (int sl = 0; sl < 2; ++sl)
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            umma_bf16_pair(tmem_base + 256u * sl, d + 2 * kk, d + (uint64_t)((1 + sl) * (kABytes >> 4) + 2 * kk), idesc1, 1u);
                } else {
                    const int k0 = 8 * (i - p.n_k);   // sixteens of activations: 8 packed columns each
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int k16 = k0 + q;
                        umma_bf16_ts_pair(tmem_base + 128u, tmem_base + (uint32_t)(k16 < 16 ? 8 * k16 : 384 + 8 * (k16 - 16)),
                                          d + (uint64_t)((1 + (q >> 2)) * (kABytes >> 4) + 2 * (q & 3)), idesc2, k16 > 0 ? 1u : 0u);
                    }
                }
                umma_commit_pair(smem_u32(empty + s));
            }
            if (ok) umma_commit_pair(smem_u32(acc2));
        }
        __syncwarp();
    } else if (warp < C::kBWarp) {
        // ===================== rows: every warp fills the stage of its number (see the layer kernel) =====================
        const RowGather g(p, lane);
        const int s = warp - C::kProdWarp0;
        const uint32_t dst0 = smem_u32(base + s * C::kStage) + (uint32_t)(g.r0 * 128);
        const TileInfo t = decode_tile(p, (int)blockIdx.x, p.sl.n_tiles);
        ChunkRows c;
        if (s < p.n_k) g.fetch(c, p, s, t);
        uint32_t ph = 0;
#pragma unroll 1
        for (int i = s; i < n_stages; i += kS) {
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(empty + s), ph ^ 1u, abort_flag))) break;
            const bool rows = i < p.n_k, gathered = rows && c.kind != SRC_DENSE;
            if (lane == 0) {
                if (rows && !gathered && c.tma_x >= 0) {
                    mbar_expect_tx(smem_u32(landed + s), (uint32_t)kABytes);
                    tma_load_2d(smem_u32(base + s * C::kStage), &tmapA, smem_u32(landed + s), c.tma_x, c.tma_y);
                } else
                    mbar_arrive(smem_u32(landed + s));
            }
            if (gathered) {
                g.copy(c, p, dst0, i == 0);
                cp_async_commit();
            }
            if (i + kS < p.n_k) g.fetch(c, p, i + kS, t);   // these loads are in flight while the copies land
            if (gathered) {
                cp_async_wait<0>();
                fence_proxy_async();   // written by cp.async (generic proxy), read by the products through the async proxy
            }
            __syncwarp();
            bool ok = true;
            if (lane == 0) {
                ok = mbar_wait(smem_u32(landed + s), ph, abort_flag);   // the stage's weights, and a dense chunk's rows
                if (ok) mbar_arrive_cluster(cluster_addr(smem_u32(full + s), 0u));
            }
            if (!__all_sync(0xffffffffu, ok)) break;
            ph ^= 1u;
        }
        cp_async_wait_all();
    } else {
        // ===================== weights (TMA): this CTA's half of every slice's rows =====================
        if (lane == 0) {
            const int half2 = mp.H2 >> 1;
#pragma unroll 1
            for (int i = 0; i < n_stages; ++i) {
                const int s = i % kS;
                if (!mbar_wait(smem_u32(empty + s), (uint32_t)((i / kS) & 1) ^ 1u, abort_flag)) break;
                const bool first = i < p.n_k;
                mbar_expect_tx(smem_u32(landed + s), first ? 2u * kABytes : 2u * (uint32_t)half2 * 128u);
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    tma_load_2d(smem_u32(base + s * C::kStage + (1 + q) * kABytes), first ? &tmapW1 : &tmapW2, smem_u32(landed + s),
                                first ? 64 * i : 64 * (2 * (i - p.n_k) + q), first ? 256 * q + 128 * rank : half2 * rank);
            }
        }
        __syncwarp();
    }

    // ---- teardown: everybody arrives here, also after an abort; neither CTA leaves while the other may still reach it
    if (*abort_flag) {
        if (tid == 0) atomicOr(p.sl.status, AIF_STATUS_TIMEOUT);
        // let copies and MMAs that are still in flight land before shared memory and TMEM go away
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == C::kMmaWarp) tmem_dealloc_pair(tmem_base, 512);
}

// The tile of a block in the kernels below, from the request table.
struct BlockTile {
    int slot, cnt;
    int64_t pos0;
};
__device__ __forceinline__ BlockTile block_tile(const ScoreLaunch &sl, int tile, int mini_batch)
{
    const ReqDev rq = find_request(sl, tile);
    int start, cnt;
    tile_range(tile - rq.tile_begin, rq.n, kTcTile, mini_batch, start, cnt);
    return BlockTile{rq.slot, cnt, rq.off + start};
}

// v_bea = w^ V (Algorithm 1 line 4) for half a tile of candidates per block: n d fused multiply-adds against 2 d bytes written
// per candidate, so memory and latency bound, and all of it independent.  V goes to shared memory once per block, the ids and
// weight rows of the 64 candidates are fetched side by side, then a thread owns eight columns (one 16-byte store) of every
// 2048 / d-th candidate.  A warp per candidate, its loads one after the other and in line with the other blocks of the
// interaction kernel, took 35 us for 9877 candidates at d = 128, n = 8.
constexpr int kBeaRows = 64;
__global__ void __launch_bounds__(256) k_bea_x(ModelDev md, ScoreLaunch sl, __nv_bfloat16 *X, int x_stride, int col)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int d = md.d, nb = md.n_bridge, tid = threadIdx.x;
    __nv_bfloat16 *V = reinterpret_cast<__nv_bfloat16 *>(smem_raw);          // [nb][d]
    float *w = reinterpret_cast<float *>(smem_raw + (size_t)nb * d * 2);     // [kBeaRows][nb]
    if (!sl.late) grid_dep_wait();
    grid_dep_launch();
    const BlockTile t = block_tile(sl, blockIdx.x, md.mini_batch);
    const int first = blockIdx.y * kBeaRows, cnt = min(kBeaRows, t.cnt - first);
    if (cnt <= 0) {
        if (sl.late && (blockIdx.x | blockIdx.y) == 0) grid_dep_wait();
        return;
    }
    const int64_t pos0 = t.pos0 + first;
    const uint4 *Vg = reinterpret_cast<const uint4 *>(sl.slots[t.slot].V);
    for (int i = tid; i < nb * d / 8; i += 256) reinterpret_cast<uint4 *>(V)[i] = Vg[i];
    for (int i = tid; i < cnt * nb; i += 256) {
        const int c = i / nb, id = sl.ids[pos0 + c];
        const bool good = id >= 0 && (int64_t)id < md.M;   // an id outside the table: zero columns
        w[i] = good ? to_f(reinterpret_cast<const __nv_bfloat16 *>(md.bea_w)[(size_t)id * nb + (i - c * nb)]) : 0.f;
    }
    __syncthreads();
    const int per_row = d / 8;
    for (int i = tid; i < cnt * per_row; i += 256) {
        const int c = i / per_row, k = (i - c * per_row) * 8;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int b = 0; b < nb; ++b) {
            const float wb = w[c * nb + b];
            const uint4 v = *reinterpret_cast<const uint4 *>(V + b * d + k);
            const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(h[q]);
                acc[2 * q] = fmaf(wb, f.x, acc[2 * q]), acc[2 * q + 1] = fmaf(wb, f.y, acc[2 * q + 1]);
            }
        }
        uint4 o;
        __nv_bfloat162 *oh = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
        for (int q = 0; q < 4; ++q) oh[q] = __floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]);
        *reinterpret_cast<uint4 *>(X + (size_t)(pos0 + c) * x_stride + col + k) = o;
    }
    if (sl.late && (blockIdx.x | blockIdx.y) == 0) grid_dep_wait();
}

// ---- interaction blocks that feed dense columns (CUDA cores; one warp per candidate) ---------------------------
// Writes, per candidate position, the att, lsh_din and simtier columns of a bf16 row [ att (d) | v_bea (d) | lsh_din (d) |
// simtier (64, first n_tiers used) ] that holds only the enabled blocks (k_bea_x writes v_bea).
__global__ void __launch_bounds__(256) k_interact_x(ModelDev md, ScoreLaunch sl, __nv_bfloat16 *X, int x_stride, int att_done, int lsh_done)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *qv = reinterpret_cast<float *>(smem_raw);                         // [8][d]
    uint32_t *sigq = reinterpret_cast<uint32_t *>(qv + 8 * md.d);            // [8][8]
    int *tiers = reinterpret_cast<int *>(sigq + 64);                         // [8][16]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d = md.d, dq = d >> 5;
    grid_dep_launch();
    grid_dep_wait();
    const BlockTile tile = block_tile(sl, blockIdx.x, md.mini_batch);
    const int cnt = tile.cnt;
    if (cnt <= 0) return;
    const int64_t pos0 = tile.pos0;
    const SlotDev slot = sl.slots[tile.slot];
    // att_done / lsh_done: those columns were already written by the tensor-core attention / LSH kernels
    const bool has_att = md.blocks & AIF_BLK_ATT, do_att = has_att && !att_done, has_bea = md.blocks & AIF_BLK_BEA;
    const bool has_din = md.blocks & AIF_BLK_LSH_DIN, has_tier = md.blocks & AIF_BLK_SIMTIER;
    const bool do_din = has_din && !lsh_done, do_tier = has_tier && !lsh_done, do_lsh = do_din || do_tier;
    const int col_din = (has_att ? d : 0) + (has_bea ? d : 0), col_tier = col_din + (has_din ? d : 0);
    using T = __nv_bfloat16;
    for (int c = warp; c < cnt; c += 8) {
        const int64_t pos = pos0 + c;
        const int id = sl.ids[pos];
        T *xrow = X + (size_t)pos * x_stride;
        if (id < 0 || (int64_t)id >= md.M) {
            // zero the columns this kernel owns; the tensor-core kernels zero theirs
            const __nv_bfloat16 z = __float2bfloat16_rn(0.f);
            for (int k = lane; k < d; k += 32) {
                if (do_att) xrow[k] = z;
                if (do_din) xrow[col_din + k] = z;
            }
            if (do_tier)
                for (int k = lane; k < 64; k += 32) xrow[col_tier + k] = z;
            continue;
        }
        const T *e = reinterpret_cast<const T *>(md.E) + (size_t)id * d;
        for (int k = lane; k < d; k += 32) qv[warp * d + k] = to_f(e[k]);
        if (do_lsh && lane < (md.lsh_bits >> 5))
            sigq[warp * 8 + lane] = reinterpret_cast<const uint32_t *>(md.sig + (size_t)id * (md.lsh_bits >> 3))[lane];
        if (lane < 16) tiers[warp * 16 + lane] = 0;
        __syncwarp();
        float att[8], din[8];
        if (do_att || do_lsh)
            warp_interact<T>(qv + warp * d, reinterpret_cast<const T *>(slot.S), slot.L, d, rsqrtf((float)d), do_att, do_lsh,
                             do_tier, sigq + warp * 8, slot.sigS, md.lsh_bits, md.n_tiers, tiers + warp * 16, att, din);
        if (do_att) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < dq) xrow[lane + 32 * q] = __float2bfloat16_rn(att[q]);
        }
        if (do_din) {
            const float nrm = md.lsh_din_norm == AIF_NORM_MEAN ? 1.0f / (float)slot.L : 1.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < dq) xrow[col_din + lane + 32 * q] = __float2bfloat16_rn(din[q] * nrm);
        }
        if (do_tier) {
            __syncwarp();
            const float nrm = md.simtier_norm == AIF_NORM_MEAN ? 1.0f / (float)slot.L : 1.0f;
            for (int k = lane; k < 64; k += 32)
                xrow[col_tier + k] = __float2bfloat16_rn(k < md.n_tiers ? (float)tiers[warp * 16 + k] * nrm : 0.f);
        }
        __syncwarp();
    }
}

constexpr int kJoinCols = 16;
__device__ __forceinline__ void join_tile(const JoinParams &p, const KeyTile &t, int y)
{
    if (t.n_parts < 2) return;   // one key block in the whole tile: the first piece has delivered
    const int row = threadIdx.x & 127, half = threadIdx.x >> 7;
    if (row >= t.cnt) return;
    const int id = p.sl.ids[t.pos0 + row];
    const bool good = id >= 0 && (int64_t)id < p.M;   // an id outside the table: a zero row
    const SplitScratch &sp = p.sl.split;
    __nv_bfloat16 *x = p.X + (size_t)(t.pos0 + row) * p.x_stride;
    const int n = t.n_parts;
    if (p.col >= 0 && y < p.d / kJoinCols) {
        const int g0 = y * (kJoinCols / 4) + half * 2;   // two groups of four columns per thread
        const float4 *rows = reinterpret_cast<const float4 *>(sp.rows) + ((size_t)t.pslot * (p.d / 4) + g0) * 128 + row;
        const size_t piece = (size_t)(p.d / 4) * 128;
        const float *st = sp.stats + (size_t)t.pslot * 256 + row;
        float m = 0.f, l = 0.f, acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (p.attention) {
            m = -INFINITY;
            for (int q = 0; q < n; ++q) m = fmaxf(m, st[q * 256 + 128]);
        }
#pragma unroll 4
        for (int q = 0; q < n; ++q) {
            const float4 a = rows[q * piece], b = rows[q * piece + 128];
            float w = 1.f;
            if (p.attention) {
                w = fast_exp2(st[q * 256 + 128] - m);   // 1 where no piece needed a running maximum
                l = fmaf(st[q * 256], w, l);
            }
            acc[0] = fmaf(w, a.x, acc[0]), acc[1] = fmaf(w, a.y, acc[1]), acc[2] = fmaf(w, a.z, acc[2]), acc[3] = fmaf(w, a.w, acc[3]);
            acc[4] = fmaf(w, b.x, acc[4]), acc[5] = fmaf(w, b.y, acc[5]), acc[6] = fmaf(w, b.z, acc[6]), acc[7] = fmaf(w, b.w, acc[7]);
        }
        // (no weight at all, every score minus infinity: no number, as in a tile that is not split)
        const float scale = p.attention ? 1.0f / l : p.row_scale * (p.row_mean ? 1.0f / (float)t.L_tile : 1.0f);
        uint4 o;
        __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(good ? acc[2 * i] * scale : 0.f, good ? acc[2 * i + 1] * scale : 0.f);
        *reinterpret_cast<uint4 *>(x + p.col + g0 * 4) = o;
    } else {
        // 64 columns of tier counts, the first n_tiers used: half 0 the first 32, half 1 the rest (zero)
        const float nrm = p.tier_mean ? 1.0f / (float)t.L_tile : 1.0f;
        const int32_t *c = sp.tiers + (size_t)t.pslot * 16 * 128 + row;
        uint4 o[4];
        __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(o);
#pragma unroll
        for (int i = 0; i < 16; ++i) h[i] = __floats2bfloat162_rn(0.f, 0.f);
        if (half == 0 && good) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                int a = 0, b = 0;
                if (2 * i < p.n_tiers)
                    for (int q = 0; q < n; ++q) a += c[(q * 16 + 2 * i) * 128], b += c[(q * 16 + 2 * i + 1) * 128];
                h[i] = __floats2bfloat162_rn((float)a * nrm, 2 * i + 1 < p.n_tiers ? (float)b * nrm : 0.f);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4 *>(x + p.x_tier + half * 32 + i * 8) = o[i];
    }
}

// Puts the pieces of split tiles together, in their order: an item is sixteen columns of a tile's rows or (SimTier on) its tier
// counts.  The pieces' sums are joined by a launch of their own and not by whichever piece comes last: a tile's records are
// 64 KB per piece, and one SM takes in 59 bytes per clock (8 pieces: 9 k cycles at the end of the launch, eq. 2's attention over
// 1000 items 13.7 -> 23 us); here a tile is read by as many SMs as there are columns to share out.
__global__ void __launch_bounds__(256) k_join_pieces(const JoinParams p)
{
    if (!p.sl.late) grid_dep_wait();
    grid_dep_launch();
    const int n_y = (p.col >= 0 ? p.d / kJoinCols : 0) + (p.x_tier >= 0 ? 1 : 0);
    const int n_items = (p.sl.jobs ? p.sl.n_jobs_dev[1] : p.sl.n_tiles) * n_y;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int tile = item / n_y, y = item - tile * n_y, job = p.sl.jobs ? p.sl.joins[tile] : tile * p.sl.parts;
        join_tile(p, p.d == 128 ? key_tile<128, true>(p.sl, job, p.mini_batch) : key_tile<64, true>(p.sl, job, p.mini_batch), y);
    }
    if (p.sl.late && blockIdx.x == 0) grid_dep_wait();
}

// Self-test of the bounded wait: one thread waits, with a short limit, on an mbarrier that nobody arrives on.  The wait
// gives up, raises the status bit and the kernel returns normally: this is the path a scoring kernel takes when a
// producer never delivers, exercised without any fault.
__global__ void k_wait_selftest(uint32_t *status, long long limit_cycles)
{
    __shared__ uint64_t bar;
    __shared__ uint32_t abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const bool done = mbar_try_wait(smem_u32(&bar), 0u, 1000u) || mbar_wait_slow(smem_u32(&bar), 0u, &abort_flag, limit_cycles);
        if (!done && abort_flag) atomicOr(status, AIF_STATUS_TIMEOUT);
    }
}

// W1 [H1 x Din] -> [H1 x k1pad]: user columns dropped, zero padding at the end.
__global__ void k_pack_w1(const __nv_bfloat16 *W1, __nv_bfloat16 *out, int H1, int din, int d, int k1, int k1pad)
{
    const int64_t total = (int64_t)H1 * k1pad;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(i / k1pad), c = (int)(i - (int64_t)j * k1pad);
        out[i] = c < k1 ? W1[(size_t)j * din + d + c] : __float2bfloat16_rn(0.f);
    }
}

// ---- host side ------------------------------------------------------------------------------------------------
struct TcPlan {
    int n_layers = 0;
    int k1 = 0, k1pad = 0, x_cols = 0;
    int n_k[kMaxHidden] = {}, n_cols[kMaxHidden] = {}, n_nchunks[kMaxHidden] = {};
    ChunkSrc src0[kMaxChunks] = {};
    CUtensorMap tmap[kMaxHidden];
    CUtensorMap tmap_half[kMaxHidden];   // the same weights, boxes of half a slice's rows (layer kernel)
    CUtensorMap tmap_quarter;            // the second layer's, boxes of a quarter of its units (small-request kernel)
    size_t cap_rows = 0;                 // rows of the context's own scratch arrays
    __nv_bfloat16 *W[kMaxHidden] = {};
    __nv_bfloat16 *H[kMaxHidden] = {};   // activations after layer k (k < last)
    __nv_bfloat16 *X = nullptr;
    uint16_t *xb = nullptr;              // cross-feature buckets [positions x F]
    TileDev *tiles = nullptr;            // tile table of a launch over several requests
    size_t tiles_cap = 0;                // its entries
    bool maps_ready = false;
};

// Slices of a layer's outputs: 256 wide, a narrower layer rounded up to a multiple of 64.
int slice_cols(int H) { return H <= 256 ? (H + 63) / 64 * 64 : 256; }

// Launches the layer kernel over a launch's tiles: persistent, one pair of CTAs per two SMs.
cudaError_t launch_layer(const LayerParams &p, int n_tiles, const CUtensorMap &tb, const CUtensorMap &to, const CUtensorMap &ta, cudaStream_t st)
{
    const int items = (n_tiles + 1) / 2 * p.n_nchunks;
    const cudaError_t e = launch_pdl_pair(k_layer_pair, dim3(2 * (items < 74 ? items : 74)), dim3(PairCfg::kThreads), PairCfg::kSmem, st, tb, to, ta, p);
    count_launch();
    return e;
}

int dense_cols(const aif_config &c)
{
    int x = 0;
    if (c.blocks & AIF_BLK_ATT) x += c.d;
    if (c.blocks & AIF_BLK_BEA) x += c.d;
    if (c.blocks & AIF_BLK_LSH_DIN) x += c.d;
    if (c.blocks & AIF_BLK_SIMTIER) x += 64;
    return x;
}

}  // namespace

bool tc_supported(const aif_config &c)
{
    if (c.dtype != AIF_BF16 || c.d % 64 != 0) return false;
    if ((uint64_t)c.M * (uint64_t)c.d * 2 / 16 >= (1ull << 32)) return false;        // row offsets are 32-bit, in 16-byte units
    if ((uint64_t)(c.max_batch_candidates + kTcTile) * 4096 / 16 >= (1ull << 32)) return false;   // same for dense rows
    if (c.blocks & AIF_BLK_CROSS) {
        if ((c.F * c.dc) % 64 != 0 || c.dc % 8 != 0 || c.B >= 65535) return false;
        if (64 % c.dc != 0 && c.dc % 64 != 0) return false;
    }
    for (int k = 0; k < c.n_hidden; ++k) {
        const int H = c.hidden[k];
        if (H <= 256 ? H % 16 != 0 : H % 256 != 0) return false;
        if (k + 1 < c.n_hidden && H % 64 != 0) return false;
    }
    if (c.hidden[c.n_hidden - 1] > 256) return false;
    aif_config tmp = c;
    const int k1 = aif_input_width(&tmp) - c.d;
    if ((k1 + 63) / 64 > kMaxChunks) return false;
    return encode_fn() != nullptr;
}

int tc_tiles_for(const aif_ctx *ctx, int n) { return tiles_of(n, kTcTile, ctx->cfg.mini_batch); }

size_t tc_tile_capacity(const aif_ctx *ctx) { return reinterpret_cast<const TcPlan *>(ctx->tc_plan)->tiles_cap; }

static TcPlan *plan_of(const aif_ctx *ctx) { return reinterpret_cast<TcPlan *>(ctx->tc_plan); }

// Allocates the tensor-path buffers (called from aif_create through tc_prepare_context).
cudaError_t tc_prepare_context(aif_ctx *ctx)
{
    const aif_config &c = ctx->cfg;
    TcPlan *pl = new TcPlan();
    ctx->tc_plan = pl;
    pl->n_layers = c.n_hidden;
    pl->k1 = ctx->input_width - c.d;
    pl->x_cols = dense_cols(c);
    // chunk list of the first layer, in the column order [e | att | cross | bea | din | simtier]
    int n = 0, xoff = 0;
    auto add = [&](int kind, int off) { pl->src0[n].kind = kind, pl->src0[n].off = off, ++n; };
    for (int o = 0; o < c.d; o += 64) add(SRC_ITEM, o * 2);
    if (c.blocks & AIF_BLK_ATT) {
        for (int o = 0; o < c.d; o += 64) add(SRC_DENSE, (xoff + o) * 2);
        xoff += c.d;
    }
    if (c.blocks & AIF_BLK_CROSS)
        for (int o = 0; o < c.F * c.dc; o += 64) add(SRC_CROSS, o);
    if (c.blocks & AIF_BLK_BEA) {
        for (int o = 0; o < c.d; o += 64) add(SRC_DENSE, (xoff + o) * 2);
        xoff += c.d;
    }
    if (c.blocks & AIF_BLK_LSH_DIN) {
        for (int o = 0; o < c.d; o += 64) add(SRC_DENSE, (xoff + o) * 2);
        xoff += c.d;
    }
    if (c.blocks & AIF_BLK_SIMTIER) add(SRC_DENSE, xoff * 2);
    pl->k1pad = n * 64;
    const size_t cap = (size_t)c.max_batch_candidates + kTcTile;
    pl->cap_rows = cap;
    auto alloc = [&](void **p, size_t bytes) -> cudaError_t {
        bytes = (bytes + 255) / 256 * 256;
        cudaError_t e = cudaMalloc(p, bytes);
        if (e != cudaSuccess) return e;
        ctx->allocations.push_back(*p);
        ctx->device_bytes += (int64_t)bytes;
        return cudaMemset(*p, 0, bytes);
    };
    cudaError_t e;
    int in_w = pl->k1pad;
    for (int k = 0; k < c.n_hidden; ++k) {
        const int H = c.hidden[k];
        pl->n_k[k] = in_w / 64;
        pl->n_cols[k] = slice_cols(H);
        pl->n_nchunks[k] = (H + pl->n_cols[k] - 1) / pl->n_cols[k];
        if ((e = alloc((void **)&pl->W[k], (size_t)H * in_w * 2)) != cudaSuccess) return e;
        if (k + 1 < c.n_hidden && (e = alloc((void **)&pl->H[k], cap * H * 2)) != cudaSuccess) return e;
        in_w = H;
    }
    if (pl->x_cols && (e = alloc((void **)&pl->X, cap * pl->x_cols * 2)) != cudaSuccess) return e;
    if ((c.blocks & AIF_BLK_CROSS) && (e = alloc((void **)&pl->xb, cap * c.F * 2)) != cudaSuccess) return e;
    {
        // Tiles never straddle a mini-batch, so every mini-batch rounds up by itself: a mini-batch of mb candidates is
        // ceil(mb / 128) tiles, and the tail of every request adds at most as many again.
        const size_t mb = (size_t)c.mini_batch;
        const size_t tpm = mb ? (mb + kTcTile - 1) / kTcTile : 0;
        const size_t body = mb ? ((size_t)c.max_batch_candidates / mb + 1) * tpm : (size_t)c.max_batch_candidates / kTcTile + 1;
        pl->tiles_cap = body + (size_t)c.max_user_states * (mb ? tpm : 1) + 64;
        if ((e = alloc((void **)&pl->tiles, pl->tiles_cap * sizeof(TileDev))) != cudaSuccess) return e;
    }
    e = cudaFuncSetAttribute(k_layer_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairCfg::kSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MlpCfg::kSmem);
    if (e != cudaSuccess) return e;
    // tensor maps over the packed weights: [H x in_w] bf16, box = 64 columns x n_cols rows, 128-byte swizzle
    EncodeFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    in_w = pl->k1pad;
    for (int k = 0; k < c.n_hidden; ++k) {
        const cuuint64_t dims[2] = {(cuuint64_t)in_w, (cuuint64_t)c.hidden[k]};
        const cuuint64_t strides[1] = {(cuuint64_t)in_w * 2};
        const cuuint32_t estr[2] = {1, 1};
        for (int half = 0; half < 2; ++half) {   // whole slices (single-launch kernel) and halves (layer kernel)
            const cuuint32_t box[2] = {64, (cuuint32_t)pl->n_cols[k] >> half};
            CUresult r = enc(half ? &pl->tmap_half[k] : &pl->tmap[k], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, pl->W[k], dims, strides, box, estr,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
        }
        if (k == 1 && tc_fused_supported(c)) {
            const cuuint32_t box[2] = {64, (cuuint32_t)c.hidden[1] / 4};
            if (enc(&pl->tmap_quarter, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, pl->W[k], dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
        }
        in_w = c.hidden[k];
    }
    pl->maps_ready = true;
    // Records of partial results, as many as a launch of this context can use: none where a sequence is one key block, no more than
    // its tiles have pieces (a context that only holds a table needs none).  64 KB each at d = 128, written before they are read, so
    // never cleared.  Splitting is for speed only: where there is no room for the records the context does without.
    auto take_split = [&](SplitScratch &sp, int64_t slots, bool tiers) -> bool {
        if (slots < 2) return true;
        const size_t bytes[3] = {(size_t)slots * 128 * c.d * 4, (size_t)slots * 256 * 4, tiers ? (size_t)slots * 16 * 128 * 4 : 0};
        void *q[3] = {};
        bool ok = true;
        for (int i = 0; i < 3; ++i) ok = ok && (bytes[i] == 0 || cudaMalloc(&q[i], bytes[i]) == cudaSuccess);
        if (!ok) {
            for (int i = 0; i < 3; ++i)
                if (q[i]) cudaFree(q[i]);
            cudaGetLastError();
            return false;
        }
        for (int i = 0; i < 3; ++i)
            if (q[i]) ctx->allocations.push_back(q[i]), ctx->device_bytes += (int64_t)bytes[i];
        sp.rows = (float *)q[0], sp.stats = (float *)q[1], sp.tiers = (int32_t *)q[2], sp.slots = (int32_t)slots;
        return true;
    };
    const int bn = c.d == 128 ? 128 : 64, key_blocks = (c.L_max + bn - 1) / bn, most = key_blocks < kMaxParts ? key_blocks : kMaxParts;
    auto records = [&](int64_t tiles, int cap) { return key_blocks < 2 ? 0 : tiles * most < cap ? tiles * most : (int64_t)cap; };
    // (by category: pieces of four key blocks of 128 and more, k_sim_tiles)
    const int64_t n_split = c.n_categories == 0 ? records((int64_t)pl->tiles_cap, kSplitSlots) : c.L_max > 4 * 128 ? kSplitSlots : 0;
    const bool att = tc_att_supported(c), lsh = tc_lsh_supported(c), tiers = c.blocks & AIF_BLK_SIMTIER;
    if (att || lsh) take_split(ctx->split, n_split, tiers && !att);
    if (att && lsh && !take_split(ctx->split_lsh, n_split, tiers)) ctx->split.slots = 0;   // both kernels take the same pieces
    if (att) take_split(ctx->split_user, records((c.L_max + kTcTile - 1) / kTcTile, kSplitSlotsUser), false);
    if (tc_att_supported(c) && (e = tc_att_prepare(ctx)) != cudaSuccess) return e;
    if (tc_fused_supported(c) && (e = tc_fused_prepare(ctx)) != cudaSuccess) return e;
    if (tc_fused_supported(c)) ctx->split_clusters = tc_split_prepare();
    if (tc_lsh_supported(c) && (e = tc_lsh_prepare(ctx)) != cudaSuccess) return e;
    if (tc_tiers_supported(c) && (e = tc_tiers_prepare(ctx)) != cudaSuccess) return e;
    if (tc_din_supported(c) && (e = tc_din_prepare(ctx)) != cudaSuccess) return e;
    if (c.n_categories > 0 && (e = sim_prepare(ctx)) != cudaSuccess) return e;
    return cudaSuccess;
}

// A launch takes ceil(jobs / 148) rounds of (key blocks of a job + what a job costs besides: the query gather before its first
// scores, its output), in units of a key block (0.9 us), and a split one the joining launch on top (about 5 us).  Splitting pays
// where the tiles leave SMs without work or fill the last round badly; a gain below a tenth is not worth the traffic.  Eq. 2 over
// 1000 items (8 tiles of 8 blocks) takes as long either way, which is where this line lies.
int split_parts(int n_tiles, int blocks, int slots)
{
    auto cost = [&](int parts) { return ((int64_t)n_tiles * parts + 147) / 148 * ((blocks + parts - 1) / parts + (parts > 1 ? 3 : 2)) + (parts > 1 ? 5 : 0); };
    int best = 1;
    for (int parts = 2; parts <= blocks && parts <= kMaxParts && (int64_t)n_tiles * parts <= slots; ++parts)
        if (cost(parts) < cost(best)) best = parts;
    return best > 1 && 10 * cost(best) < 9 * cost(1) ? best : 1;
}

cudaError_t launch_join_pieces(const JoinParams &p, cudaStream_t st)
{
    const int n_y = (p.col >= 0 ? p.d / kJoinCols : 0) + (p.x_tier >= 0 ? 1 : 0);
    const int items = (p.sl.jobs ? kSplitSlots / 2 : p.sl.n_tiles) * n_y, grid = items < 148 * 6 ? items : 148 * 6;
    const cudaError_t e = launch_pdl(k_join_pieces, dim3(grid), dim3(256), 0, st, p);
    count_launch();
    return e;
}

const void *tc_weight_half_tmap(const aif_ctx *ctx, int k) { return &plan_of(ctx)->tmap_half[k]; }
const void *tc_weight_quarter_tmap(const aif_ctx *ctx) { return &plan_of(ctx)->tmap_quarter; }
const void *tc_weight_tmap(const aif_ctx *ctx, int k) { return &plan_of(ctx)->tmap[k]; }

void tc_destroy_context(aif_ctx *ctx)
{
    if (ctx->tc_att_plan) tc_att_destroy(ctx);
    if (ctx->tc_lsh_plan) tc_lsh_destroy(ctx);
    if (ctx->tc_tier_plan) tc_tiers_destroy(ctx);
    if (ctx->tc_din_plan) tc_din_destroy(ctx);
    delete plan_of(ctx);
    ctx->tc_plan = nullptr;
}

cudaError_t tc_prepare_weights(aif_ctx *ctx, const aif_weights *w, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    TcPlan *pl = plan_of(ctx);
    k_pack_w1<<<296, 256, 0, st>>>((const __nv_bfloat16 *)w->W[0], pl->W[0], c.hidden[0], ctx->input_width, c.d, pl->k1,
                                   pl->k1pad);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    for (int k = 1; k < c.n_hidden; ++k) {
        e = cudaMemcpyAsync(pl->W[k], w->W[k], (size_t)c.hidden[k] * c.hidden[k - 1] * 2, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_wait_selftest(const aif_ctx *ctx, long long limit_cycles, cudaStream_t st)
{
    k_wait_selftest<<<1, 32, 0, st>>>(ctx->status, limit_cycles);
    count_launch();
    return cudaGetLastError();
}

size_t tc_scratch_row_bytes(const aif_ctx *ctx)
{
    const aif_config &c = ctx->cfg;
    size_t cols = (size_t)plan_of(ctx)->x_cols;
    for (int k = 0; k + 1 < c.n_hidden; ++k) cols += (size_t)c.hidden[k];
    if (c.blocks & AIF_BLK_CROSS) cols += (size_t)c.F;
    return cols * 2;
}

void tc_scratch_layout(const aif_ctx *ctx, void *base, size_t rows, TcScratch *out)
{
    const aif_config &c = ctx->cfg;
    unsigned char *p = reinterpret_cast<unsigned char *>(base);
    out->X = p;
    p += rows * (size_t)plan_of(ctx)->x_cols * 2;
    for (int k = 0; k < kMaxHidden; ++k) {
        out->H[k] = nullptr;
        if (k + 1 < c.n_hidden) {
            out->H[k] = p;
            p += rows * (size_t)c.hidden[k] * 2;
        }
    }
    out->xb = (c.blocks & AIF_BLK_CROSS) ? p : nullptr;
    out->tiles = nullptr;
    out->split = false;
    out->rows = rows;
}

// One dense layer over `rows` consecutive rows of a row-major bf16 matrix, with the layer kernel: out = act(A W^T + b)
// (bf16), or the packed sign bits of A W^T.  Used by the item side of the nearline pipeline.
cudaError_t tc_dense_layer(const aif_ctx *ctx, const DenseLayer &L, int64_t rows, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    EncodeFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    LayerParams p{};
    p.sl.slots = ctx->slots_dev, p.sl.reqs = nullptr, p.sl.n_req = 1;
    p.sl.single = ReqDev{0, (int32_t)rows, 0, 0, 0};
    p.sl.n_tiles = (int32_t)((rows + kTcTile - 1) / kTcTile), p.sl.total = rows, p.sl.max_L = 0;
    p.sl.ids = nullptr, p.sl.logits = nullptr, p.sl.status = ctx->status, p.sl.late = L.late;
    p.n_cols = slice_cols(L.H), p.n_nchunks = (L.H + p.n_cols - 1) / p.n_cols, p.n_out = L.H, p.n_k = L.in_w / 64, p.mini_batch = 0;
    p.E = (const uint8_t *)ctx->E, p.M = ctx->cfg.M, p.e_row_bytes = ctx->cfg.d * 2;
    p.X = (const uint8_t *)L.A;
    p.B = 1, p.dc = 8, p.F = 0, p.xb = nullptr, p.check_ids = 0;
    for (int i = 0; i < p.n_k; ++i) p.src[i].kind = SRC_DENSE, p.src[i].off = i * 128;
    p.epi = L.sign_bits ? EPI_SIGN : EPI_STORE;
    p.bias_from_slot = 0, p.bias = L.bias, p.emit_sigmoid = 0, p.linear_out = L.relu ? 0 : 1;
    p.out = (__nv_bfloat16 *)L.out, p.out_stride = L.H, p.sig_out = (uint8_t *)L.out;
    p.w_out = nullptr, p.b_out = nullptr;
    const cuuint32_t estr[2] = {1, 1};
    CUtensorMap tmap_b, tmap_a, tmap_out;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)L.in_w, (cuuint64_t)L.H};
        const cuuint64_t strides[1] = {(cuuint64_t)L.in_w * 2};
        const cuuint32_t box[2] = {64, (cuuint32_t)p.n_cols / 2};
        if (enc(&tmap_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(L.W), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[2] = {(cuuint64_t)L.in_w, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)L.in_w * 2};
        const cuuint32_t box[2] = {64, 128};
        if (enc(&tmap_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(L.A), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    tmap_out = tmap_b;
    if (!L.sign_bits) {
        const cuuint64_t dims[2] = {(cuuint64_t)L.H, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)L.H * 2};
        const cuuint32_t box[2] = {32, 32};
        if (enc(&tmap_out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, L.out, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    return launch_layer(p, p.sl.n_tiles, tmap_b, tmap_out, tmap_a, st);
}

cudaError_t launch_score_tc(const aif_ctx *ctx, const ScoreLaunch &sl, int64_t, cudaStream_t st)
{
    TcPlan *pl = plan_of(ctx);
    TcScratch sc;
    sc.X = pl->X;
    sc.xb = pl->xb;
    sc.tiles = pl->tiles;
    sc.split = true;
    sc.rows = pl->cap_rows;
    for (int k = 0; k < kMaxHidden; ++k) sc.H[k] = pl->H[k];
    return launch_score_tc_scratch(ctx, sl, st, sc);
}

cudaError_t launch_score_tc_scratch(const aif_ctx *ctx, const ScoreLaunch &sl_in, cudaStream_t st, const TcScratch &sc)
{
    if (sl_in.n_tiles <= 0) return cudaSuccess;
    ScoreLaunch sl = sl_in;
    sl.tiles = nullptr;
    if (sc.split) sl.split = ctx->split;
    const aif_config &c = ctx->cfg;
    TcPlan *pl = plan_of(ctx);
    const ModelDev md = make_model(ctx);
    timing_begin(ctx, st);
    // a launch that fits the machine in one round of tiles: the whole pass in one kernel, one CTA per tile
    if (c.n_categories == 0 && sl.n_tiles <= kFusedMaxTiles && sl.max_L <= 256 && tc_fused_supported(c)) {
        StageRange range("aif score_fused");
        const int tile = sl.reqs ? 0 : tc_split_tile(ctx, sl.single.n, st);
        cudaError_t e = tile ? launch_request_split(ctx, sl, tile, st) : launch_request_fused(ctx, sl, st);
        timing_mark(ctx, tile ? "score_split" : "score_fused", st);
        return e;
    }
    // ids across the bus: on the way through the bucket kernel where that one comes first, else by a copy of their own
    if (sl.ids_copy && (c.n_categories > 0 || !(c.blocks & AIF_BLK_CROSS))) {
        cudaError_t e = launch_stage_ids(sl.ids, sl.ids_copy, sl.total, st);
        if (e != cudaSuccess) return e;
        sl.ids = sl.ids_copy, sl.ids_copy = nullptr;
    }
    SimPlace place{};
    if (c.n_categories > 0) {
        // candidates grouped by (request, category): tiles, grouped ids and the way back to the caller's order
        if (sc.rows < (size_t)sl.total + kTcTile || !ctx->sim_plan) return cudaErrorInvalidValue;
        StageRange range("aif group");
        cudaError_t e = sim_group_candidates(ctx, sl, place, sl.reqs ? (TileDev *)sc.tiles : nullptr, st);
        timing_mark(ctx, "group", st);
        if (e != cudaSuccess) return e;
    } else if (sl.reqs && sc.tiles) {   // several requests: look every tile up once
        cudaError_t e = launch_pdl(k_tile_table, dim3((sl.n_tiles + 255) / 256), dim3(256), 0, st, sl, c.mini_batch, (TileDev *)sc.tiles);
        count_launch();
        if (e != cudaSuccess) return e;
        sl.tiles = (const TileDev *)sc.tiles;
    }
    const int F = (c.blocks & AIF_BLK_CROSS) ? c.F : 0;
    auto buckets = [&](int late) -> cudaError_t {
        if (F == 0 && !place.where) return cudaSuccess;
        StageRange range("aif buckets");
        const int64_t n = sl.total;   // a warp per 32 candidates
        const int grid = (int)((n + 255) / 256 < 148 * 16 ? (n + 255) / 256 : 148 * 16);
        // launches that leave SMs without a block split the fields of a candidate over up to eight warps, except where a read
        // of the ids crosses the bus
        const int rounds = F == 0 ? 1 : F & 1 ? F : F / 2, want_y = sl.ids_copy ? 1 : 296 / grid;
        const int grid_y = want_y < 1 ? 1 : want_y > 8 ? (rounds < 8 ? rounds : 8) : want_y > rounds ? rounds : want_y;
        auto kernel = (c.B & (c.B - 1)) == 0 ? k_cross_buckets<true> : k_cross_buckets<false>;
        cudaError_t e = launch_pdl(kernel, dim3(grid, grid_y), dim3(256), 0, st, sl.ids, sl.total, c.M, F, c.B, c.B > 0 ? ~0ull / (uint64_t)c.B : 0ull, c.bucket_mode, (uint16_t *)sc.xb, sl.ids_copy, place, late);
        if (sl.ids_copy) sl.ids = sl.ids_copy;
        if (place.where) sl.ids = place.ids;
        count_launch();
        timing_mark(ctx, "buckets", st);
        return e;
    };
    const bool att_tc = ctx->tc_att_plan != nullptr;
    const int lsh_blocks = c.blocks & (AIF_BLK_LSH_DIN | AIF_BLK_SIMTIER);
    const bool lsh_tc = lsh_blocks && ctx->tc_lsh_plan != nullptr;
    // Attention, bridge columns, LSH and buckets need nothing of each other: behind the first one the others run beside it, on the SMs
    // it leaves idle (78 tiles are 78 CTAs of an attention kernel that fills an SM with one) and in its tail.  The buckets come
    // first where they bring the ids.
    const bool buckets_first = place.where || sl.ids_copy || !(att_tc || lsh_tc);
    cudaError_t eb = buckets_first ? buckets(0) : cudaSuccess;
    if (eb != cudaSuccess) return eb;
    // What does not depend on the category takes the grouped candidates request by request, in whole tiles: the groups of a request
    // are its positions, in another order.  By the groups' tiles the layers ran on rows that were mostly padding (20 candidates per
    // category: 800 tiles instead of 130).
    ScoreLaunch sl_rows = sl;
    if (c.n_categories > 0) sl_rows.n_tiles = sl_in.n_tiles, sl_rows.tiles = sl.reqs ? (const TileDev *)sc.tiles : nullptr;
    // few tiles with many keys: their keys over several CTAs each (the table of jobs does it where categories are on)
    // LSH-DIN through sums of the request's own, where that is the shorter way; SimTier then counts by itself.  The sums come first and
    // need nothing of the call: what follows runs beside them.
    const bool din = c.blocks & AIF_BLK_LSH_DIN, tier = c.blocks & AIF_BLK_SIMTIER;
    const bool din_sums = lsh_tc && din && sc.split && (!tier || ctx->tc_tier_plan) && tc_din_pays(ctx, sl);
    // (never slower than the pass that could also do eq. 8, us of the call, c2's shape without attention: 100 candidates of 50 keys 21.4 / 23.0, 1000 of
    // 1000 23.2 / 28.6, 64 x 5000 of 200 408 / 435, 2 x 5000 of 20 000 by 100 categories 53.8 / 57.8; d = 256, 100 of 50 33.4 / 36.1)
    const bool tiers_alone = tier && ctx->tc_tier_plan && (din_sums || !din);
    int late = 0;
    if (din_sums) {
        StageRange range("aif lsh sums");
        ScoreLaunch sl_sums = sl;
        sl_sums.late = buckets_first;
        const cudaError_t e = launch_din_sums(ctx, sl_sums, 0, st);
        timing_mark(ctx, "lsh_sums", st);
        if (e != cudaSuccess) return e;
        late = !buckets_first;   // (ids that the buckets bring are waited for)
    }
    if (!sl.jobs) sl.parts = split_parts(sl.n_tiles, (sl.max_L + (c.d == 128 ? 127 : 63)) / (c.d == 128 ? 128 : 64), sl.split.slots);
    JoinParams join_att{}, join_lsh{};
    if (att_tc) {
        StageRange range("aif attention");
        ScoreLaunch sl_att = sl;
        sl_att.late = late;
        cudaError_t e = launch_att_tc(ctx, sl_att, st, sc.X, pl->x_cols, sc.rows, join_att);
        timing_mark(ctx, "attention", st);
        if (e != cudaSuccess) return e;
    }
    if (att_tc) late = 1;
    auto bea = [&]() -> cudaError_t {
        if (!(c.blocks & AIF_BLK_BEA)) return cudaSuccess;
        StageRange range("aif bea");
        ScoreLaunch sl_bea = sl_rows;
        sl_bea.late = late;
        const size_t smem = (size_t)c.n_bridge * c.d * 2 + (size_t)kBeaRows * c.n_bridge * 4;
        cudaError_t e = launch_pdl(k_bea_x, dim3(sl_rows.n_tiles, kTcTile / kBeaRows), dim3(256), smem, st, md, sl_bea, (__nv_bfloat16 *)sc.X, pl->x_cols,
                                   (c.blocks & AIF_BLK_ATT) ? c.d : 0);
        count_launch();
        timing_mark(ctx, "bea", st);
        return e;
    };
    if (att_tc && (eb = bea()) != cudaSuccess) return eb;
    // columns of X: [ att | v_bea | lsh_din | simtier (64) ], enabled blocks only
    const int x_lsh = ((c.blocks & AIF_BLK_ATT) ? c.d : 0) + ((c.blocks & AIF_BLK_BEA) ? c.d : 0);
    const int x_din = din ? x_lsh : -1, x_tier = tier ? x_lsh + (din ? c.d : 0) : -1;
    if (lsh_tc && !(din_sums && !tier)) {
        StageRange range("aif lsh");
        ScoreLaunch sl_lsh = sl;
        sl_lsh.late = late;
        if (att_tc && sc.split) sl_lsh.split = ctx->split_lsh;   // records of its own: the attention's are not joined yet
        cudaError_t e = tiers_alone ? launch_tiers(ctx, sl_lsh, st, sc.X, pl->x_cols, x_tier, join_lsh)
                                    : launch_lsh_tc(ctx, sl_lsh, st, sc.X, pl->x_cols, sc.rows, x_din, x_tier, join_lsh);
        timing_mark(ctx, din_sums ? "simtier" : "lsh", st);
        if (e != cudaSuccess) return e;
        late = 1;
    }
    // the pieces of keys: the first join waits for both kernels, the second one runs beside it
    join_att.sl.late = 0;
    if (join_att.d && (eb = launch_join_pieces(join_att, st)) != cudaSuccess) return eb;
    if (join_lsh.d) {
        join_lsh.sl.late = join_att.d != 0;
        if ((eb = launch_join_pieces(join_lsh, st)) != cudaSuccess) return eb;
    }
    if (!buckets_first && (eb = buckets(late)) != cudaSuccess) return eb;
    if (din_sums) {
        StageRange range("aif lsh rows");
        ScoreLaunch sl_din = sl;
        sl_din.late = 0;
        cudaError_t e = cudaSuccess;
        for (int r0 = 0; e == cudaSuccess && r0 < sl.n_req; r0 += din_requests_at_once(ctx)) {   // (the first round's sums are there)
            if (r0 > 0) e = launch_din_sums(ctx, sl_din, r0, st);
            if (e == cudaSuccess) e = launch_din_apply(ctx, sl_din, r0, st, sc.X, pl->x_cols, sc.rows, x_din);
        }
        timing_mark(ctx, "lsh_rows", st);
        if (e != cudaSuccess) return e;
    }
    const bool need_att = (c.blocks & AIF_BLK_ATT) && !att_tc, need_lsh = lsh_blocks && !lsh_tc;
    if (!att_tc && (eb = bea()) != cudaSuccess) return eb;
    if (need_att || need_lsh) {
        StageRange range("aif interact");
        const size_t smem = (size_t)8 * c.d * 4 + 64 * 4 + 128 * 4;
        cudaError_t e = launch_pdl(k_interact_x, dim3(sl.n_tiles), dim3(256), smem, st, md, sl, (__nv_bfloat16 *)sc.X, pl->x_cols,
                                   att_tc ? 1 : 0, lsh_tc ? 1 : 0);
        count_launch();
        timing_mark(ctx, "interact", st);
        if (e != cudaSuccess) return e;
    }
    // two layers of 512 and at most 256 units, all tiles at once on the machine: one kernel
    const bool whole_mlp = c.n_hidden == 2 && c.hidden[0] == MlpCfg::kH1 && c.hidden[1] <= 256 && c.hidden[1] % 64 == 0 && sl_rows.n_tiles <= 148;
    static const char *names[kMaxHidden] = {"layer1", "layer2", "layer3", "layer4"};
    static const char *range_names[kMaxHidden] = {"aif layer1", "aif layer2", "aif layer3", "aif layer4"};
    for (int k = 0; k < c.n_hidden; ++k) {
        StageRange range(range_names[k]);
        LayerParams p{};
        p.sl = sl_rows;
        p.n_nchunks = pl->n_nchunks[k], p.n_cols = pl->n_cols[k], p.n_out = c.hidden[k], p.n_k = pl->n_k[k], p.mini_batch = c.mini_batch;
        p.E = (const uint8_t *)ctx->E, p.M = c.M, p.e_row_bytes = c.d * 2;
        p.B = c.B > 0 ? c.B : 1, p.dc = c.dc > 0 ? c.dc : 8, p.F = c.F, p.xb = (const uint16_t *)sc.xb;
        p.T0 = (const uint8_t *)ctx->slots[0].dev.T, p.slot_bytes = (int64_t)ctx->slot_bytes;
        p.check_ids = k == 0;
        if (k == 0) {
            p.X = (const uint8_t *)sc.X;
            for (int i = 0; i < p.n_k; ++i) p.src[i] = pl->src0[i];
        } else {
            p.X = (const uint8_t *)sc.H[k - 1];
            for (int i = 0; i < p.n_k; ++i) p.src[i].kind = SRC_DENSE, p.src[i].off = i * 128;
        }
        const bool last = k + 1 == c.n_hidden;
        // store target of the epilogue: the activation array as a [rows x hidden[k]] tensor, 32 x 32 boxes, 64-byte swizzle
        CUtensorMap tmap_out = pl->tmap[k];
        if (!last) {
            const cuuint64_t dims[2] = {(cuuint64_t)c.hidden[k], (cuuint64_t)sc.rows};
            const cuuint64_t strides[1] = {(cuuint64_t)c.hidden[k] * 2};
            const cuuint32_t box[2] = {32, 32};
            const cuuint32_t estr[2] = {1, 1};
            CUresult r = encode_fn()(&tmap_out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, sc.H[k], dims, strides, box, estr,
                                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
        }
        p.epi = last ? EPI_DOT : EPI_STORE;
        p.bias_from_slot = k == 0, p.bias = ctx->b[k], p.emit_sigmoid = c.emit_sigmoid;
        p.out = (__nv_bfloat16 *)sc.H[k], p.out_stride = c.hidden[k];
        p.w_out = (const __nv_bfloat16 *)ctx->w_out, p.b_out = ctx->b_out;
        // load source of the dense chunks: X (layer 1) or the previous activations, 64-column x 128-row tiles
        CUtensorMap tmap_a = pl->tmap[k];
        const int dense_w = k == 0 ? pl->x_cols : c.hidden[k - 1];
        if (dense_w > 0) {
            const cuuint64_t dims[2] = {(cuuint64_t)dense_w, (cuuint64_t)sc.rows};
            const cuuint64_t strides[1] = {(cuuint64_t)dense_w * 2};
            const cuuint32_t box[2] = {64, 128};
            const cuuint32_t estr[2] = {1, 1};
            CUresult r = encode_fn()(&tmap_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint8_t *>(p.X), dims, strides, box, estr,
                                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
        }
        if (whole_mlp) {
            MlpParams mp{p, c.hidden[1], ctx->b[1]};
            const cudaError_t e = launch_pdl_pair(k_mlp_pair, dim3((sl_rows.n_tiles + 1) / 2 * 2), dim3(MlpCfg::kThreads), MlpCfg::kSmem, st, tmap_a, pl->tmap_half[0],
                                                  pl->tmap_half[1], mp);
            count_launch();
            timing_mark(ctx, "mlp", st);
            return e;
        }
        const cudaError_t e = launch_layer(p, sl_rows.n_tiles, pl->tmap_half[k], tmap_out, tmap_a, st);
        timing_mark(ctx, names[k], st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace aif
