// Category sub-sequences (Section 3.3, SIM-hard): the long-term sequence is kept as <user, category, sub-sequence>, and a
// candidate interacts only with the sub-sequence of its own category.
//
// User side (in parallel with retrieval): the projected sequence and its +-1 signatures are laid out a second time,
// grouped by category, every sub-sequence starting on a multiple of 128 rows and padded with zero rows to the next one.
// This is the pre-cache of parsed sub-sequences for all of the user's categories.
//
// Real time: the candidates of a launch are grouped by (request, category); every group becomes tiles of up to 128
// candidates that carry their sub-sequence's key range, and the tensor-core kernels walk those tiles.  The number of
// tiles depends on the data, so it is left in device memory for the kernels to read; logits go back to the caller's
// order through an index.
#include "aif_device.cuh"
#include "aif_internal.h"
#include "aif_tc_ptx.cuh"

namespace aif {
namespace {

constexpr int kCatBlock = 1024;   // sequence items per block of the grouping passes

__device__ __forceinline__ int category_of(int id, int n_cat, int mode)
{
    if (mode == AIF_BUCKET_MOD) return id % n_cat;
    return (int)(mix64((uint64_t)id, (uint64_t)AIF_CATEGORY_FIELD) % (uint64_t)n_cat);
}

// ---- user side ------------------------------------------------------------------------------------------------
// hist[b][c] = items of category c among the block's 1024 sequence items
__global__ void __launch_bounds__(kCatBlock) k_cat_hist(const int32_t *__restrict__ cat, int L, int n_cat, int32_t *__restrict__ hist,
                                                        uint32_t *status)
{
    extern __shared__ int h_s[];
    for (int c = threadIdx.x; c < n_cat; c += kCatBlock) h_s[c] = 0;
    __syncthreads();
    const int j = blockIdx.x * kCatBlock + threadIdx.x;
    if (j < L) {
        const int c = cat[j];
        if (c >= 0 && c < n_cat) atomicAdd(&h_s[c], 1);
        else atomicOr(status, AIF_STATUS_BAD_ID);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < n_cat; c += kCatBlock) hist[(size_t)blockIdx.x * n_cat + c] = h_s[c];
}

// One block: hist[b][c] becomes the number of items of category c in earlier blocks; cat_len[c] the total; cat_off[c]
// the first row of the sub-sequence, sub-sequences following each other on multiples of 128 rows.
__global__ void __launch_bounds__(kCatBlock) k_cat_scan(int n_blocks, int n_cat, int32_t *__restrict__ hist, int32_t *__restrict__ cat_off,
                                                        int32_t *__restrict__ cat_len)
{
    __shared__ int32_t carry;
    __shared__ int32_t part[kCatBlock];
    for (int c = threadIdx.x; c < n_cat; c += kCatBlock) {
        int run = 0;
        for (int b = 0; b < n_blocks; ++b) {
            const int v = hist[(size_t)b * n_cat + c];
            hist[(size_t)b * n_cat + c] = run;
            run += v;
        }
        cat_len[c] = run;
    }
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    // exclusive scan of the padded lengths, 1024 categories at a time
    for (int c0 = 0; c0 < n_cat; c0 += kCatBlock) {
        const int c = c0 + threadIdx.x;
        const int v = c < n_cat ? (cat_len[c] + 127) / 128 * 128 : 0;
        part[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < kCatBlock; o <<= 1) {
            const int add = (int)threadIdx.x >= o ? part[threadIdx.x - o] : 0;
            __syncthreads();
            part[threadIdx.x] += add;
            __syncthreads();
        }
        if (c < n_cat) cat_off[c] = carry + part[threadIdx.x] - v;
        __syncthreads();
        if (threadIdx.x == kCatBlock - 1) carry += part[kCatBlock - 1];
        __syncthreads();
    }
}

// map[j] = row of sequence item j in the grouped sequence: its sub-sequence's first row + items of its category in
// earlier blocks + items of its category before it in this block (counted, not raced for: the order inside a
// sub-sequence is the order of the sequence, the same in every run).  -1 for a category outside the range.
__global__ void __launch_bounds__(kCatBlock) k_cat_place(const int32_t *__restrict__ cat, int L, int n_cat, const int32_t *__restrict__ hist,
                                                         const int32_t *__restrict__ cat_off, int32_t *__restrict__ map)
{
    __shared__ int32_t c_s[kCatBlock];
    const int j = blockIdx.x * kCatBlock + threadIdx.x;
    const int c = j < L ? cat[j] : -1;
    c_s[threadIdx.x] = c;
    __syncthreads();
    if (j >= L) return;
    if (c < 0 || c >= n_cat) {
        map[j] = -1;
        return;
    }
    int rank = 0;
    for (int i = 0; i < (int)threadIdx.x; ++i) rank += c_s[i] == c;
    map[j] = cat_off[c] + hist[(size_t)blockIdx.x * n_cat + c] + rank;
}

// dst[map[j]] = src[j], rows of row_bytes (a multiple of 16)
__global__ void __launch_bounds__(256) k_group_rows(const uint4 *__restrict__ src, const int32_t *__restrict__ map, int L, int vec_per_row,
                                                    uint4 *__restrict__ dst)
{
    const int64_t total = (int64_t)L * vec_per_row;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(i / vec_per_row), v = (int)(i - (int64_t)j * vec_per_row);
        const int r = map[j];
        if (r >= 0) dst[(int64_t)r * vec_per_row + v] = src[i];
    }
}

// ---- real time ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int request_of(const ScoreLaunch &sl, int64_t pos, ReqDev &rq)
{
    if (sl.reqs == nullptr) {
        rq = sl.single;
        return 0;
    }
    int lo = 0, hi = sl.n_req - 1;
    while (lo < hi) {   // last request that begins at or before pos (empty requests share their successor's start)
        const int mid = (lo + hi + 1) >> 1;
        if (sl.reqs[mid].off <= pos) lo = mid;
        else hi = mid - 1;
    }
    rq = sl.reqs[lo];
    return lo;
}

// group of a candidate: request index * n_cat + category (category 0 for an id outside the table: its logit is NaN anyway)
__device__ __forceinline__ int group_of(const ScoreLaunch &sl, int64_t pos, int64_t M, int n_cat, int mode, int &id_out)
{
    ReqDev rq;
    const int r = request_of(sl, pos, rq);
    const int id = sl.ids[pos];
    id_out = id;
    const int c = (id >= 0 && (int64_t)id < M) ? category_of(id, n_cat, mode) : 0;
    return r * n_cat + c;
}

// where[pos] = (group of candidate pos, its rank inside the group); the group counts.  The order inside a group is arbitrary.
// On the way, the tiles of the launch's requests as they would be without categories, for the kernels that take them so.
__global__ void __launch_bounds__(256) k_sim_count(ScoreLaunch sl, int64_t M, int n_cat, int mode, int32_t *__restrict__ grp_cnt, int2 *__restrict__ where,
                                                   int mini_batch, TileDev *__restrict__ row_tiles)
{
    grid_dep_launch();
    grid_dep_wait();
    if (row_tiles)
        for (int tile = (int)(blockIdx.x * blockDim.x + threadIdx.x); tile < sl.n_tiles; tile += (int)(gridDim.x * blockDim.x))
            row_tiles[tile] = tile_entry(sl, tile, mini_batch);
    for (int64_t pos = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; pos < sl.total; pos += (int64_t)gridDim.x * blockDim.x) {
        int id;
        const int g = group_of(sl, pos, M, n_cat, mode, id);
        where[pos] = make_int2(g, atomicAdd(&grp_cnt[g], 1));
    }
}

// One block over the groups: first grouped position of every group (exclusive scan of the counts), the jobs of the attention and
// LSH kernels, their number; the counts go back to zero for the next launch (the ranks place the candidates: k_cross_buckets).
// A group is ceil(candidates / 128) tiles.  A tile's cost is its number of key blocks, from none to hundreds (a user's favourite
// category holds a fifth of the sequence), so tiles with more than an SM's share of the launch are cut into pieces of that share
// (below); a tile left whole made the launch as long as the longest sub-sequence (150 key blocks of one tile against 22 per SM on
// average).  Jobs are laid out by size, largest first (in classes of a quarter octave), and every second row of 148 runs backwards:
// job j goes to CTA j mod 148, so the CTA with the largest job of one row gets the smallest of the next (4 x 10^4 candidates over
// 100 categories of 10^5 items, with pieces of half a share: at most 29 blocks per SM for 22 on average; 38 in plain order).
struct SimGroup {
    int32_t cnt, start, slot, len, key0, np, j0, p0;
};

__global__ void __launch_bounds__(1024) k_sim_tiles(ScoreLaunch sl, int n_groups, int n_cat, int32_t *__restrict__ grp_cnt,
                                                    int32_t *__restrict__ grp_start, JobDev *__restrict__ jobs, int job_cap,
                                                    int32_t *__restrict__ joins, int32_t *__restrict__ n_out)
{
    constexpr int kClasses = 128;
    __shared__ SimGroup grp[1024];
    __shared__ int32_t warp_sum_s[32];
    __shared__ long long warp_blocks_s[32];
    __shared__ int32_t carry_c, pslot_cur, join_cur;
    __shared__ int32_t cls_jobs[kClasses], cls_base[kClasses];
    __shared__ int32_t n_jobs_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    grid_dep_launch();
    grid_dep_wait();
    if (tid == 0) carry_c = 0, pslot_cur = 0, join_cur = 0;
    if (tid < kClasses) cls_jobs[tid] = 0;
    __syncthreads();
    auto key_blocks = [](int len) { return len > 0 ? (len + 127) / 128 : 1; };
    auto class_of = [](int blocks) {   // four classes per octave (below four blocks: one per octave)
        const int k = 31 - __clz(blocks);
        return k < 2 ? 4 * k : 4 * k + ((blocks >> (k - 2)) & 3);
    };
    // a thread per group and batch of 1024 groups; what it looked up stays with it where one batch is all there is
    SimGroup me{};
    auto look_up = [&](int g) {
        me.cnt = g < n_groups ? grp_cnt[g] : 0;
        if (me.cnt == 0) return;
        const int r = g / n_cat, c = g - r * n_cat;
        me.slot = sl.reqs ? sl.reqs[r].slot : sl.single.slot;
        const SlotDev *sd = sl.slots + me.slot;
        me.len = sd->cat_len[c], me.key0 = sd->cat_off[c];
    };
    // pass 1: grouped positions (exclusive scan of the counts) and the launch's key blocks
    long long blocks = 0;
    for (int g0 = 0; g0 < n_groups; g0 += 1024) {
        const int g = g0 + tid;
        look_up(g);
        int run = me.cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += v;
        }
        if (lane == 31) warp_sum_s[warp] = run;
        __syncthreads();
        int before = lane < warp ? warp_sum_s[lane] : 0;
        before = __reduce_add_sync(0xffffffffu, before) + carry_c;
        me.start = before + run - me.cnt;
        if (g < n_groups) grp_start[g] = me.start;
        if (me.cnt > 0) blocks += (long long)((me.cnt + kTcTile - 1) / kTcTile) * key_blocks(me.len);
        __syncthreads();
        if (tid == 1023) carry_c = me.start + me.cnt;
        __syncthreads();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) blocks += __shfl_xor_sync(0xffffffffu, blocks, o);
    if (lane == 0) warp_blocks_s[warp] = blocks;
    __syncthreads();
    blocks = warp_blocks_s[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) blocks += __shfl_xor_sync(0xffffffffu, blocks, o);
    // Key blocks of a piece.  Tiles with more are cut into ceil(blocks / piece) pieces: at most 2 blocks / piece <= kSplitSlots
    // records of partial results.  Below four blocks a piece is mostly its own start and end.
    // An SM's share of the launch is one piece: every record is 64 KB written and read again.  With pieces of half a share the two
    // joins took 26 of 212 us (4 x 10^4 candidates, 10^5 keys in 100 categories), with shares 203 us in all; with two shares to a
    // piece the longest tiles are alone at the end (215 us).
    const int piece = sl.split.slots >= kSplitSlots ? max(4, (int)((blocks + 148 - 1) / 148)) : 0x7fffffff;
    auto pieces_of = [&](int len) {
        const int nb = key_blocks(len);
        return nb > piece ? (nb + piece - 1) / piece : 1;
    };
    const bool one_batch = n_groups <= 1024;
    // pass 2: jobs per size class (a piece's share of the keys)
    for (int g0 = 0; g0 < n_groups; g0 += 1024) {
        if (!one_batch) look_up(g0 + tid);
        if (me.cnt > 0) {
            me.np = pieces_of(me.len);
            atomicAdd(&cls_jobs[class_of(key_blocks(me.len) / me.np)], (me.cnt + kTcTile - 1) / kTcTile * me.np);
        }
    }
    __syncthreads();
    if (warp == 0) {   // first job of every class, largest first
        int n[4], run = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) n[i] = cls_jobs[kClasses - 1 - 4 * lane - i], run += n[i];
        int before = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, before, o);
            if (lane >= o) before += v;
        }
        if (lane == 31) n_out[0] = n_jobs_s = min(before, job_cap);
        before -= run;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cls_base[kClasses - 1 - 4 * lane - i] = before;
            cls_jobs[kClasses - 1 - 4 * lane - i] = 0;   // from here on the class's cursor
            before += n[i];
        }
    }
    __syncthreads();
    // row j / 148 of the jobs, whole rows in turn forwards and backwards
    auto place_of = [&](int j) {
        const int row = j / 148, col = j - row * 148;
        return (row & 1) && row < n_jobs_s / 148 ? row * 148 + 147 - col : j;
    };
    // pass 3: the records, a warp per group of the batch; the counts go back to zero
    for (int g0 = 0; g0 < n_groups; g0 += 1024) {
        const int g = g0 + tid;
        if (!one_batch) {
            look_up(g);
            if (g < n_groups) me.start = grp_start[g];
        }
        if (me.cnt > 0) {
            grp_cnt[g] = 0;
            me.np = pieces_of(me.len);
            const int nt = (me.cnt + kTcTile - 1) / kTcTile, k = class_of(key_blocks(me.len) / me.np);
            me.j0 = cls_base[k] + atomicAdd(&cls_jobs[k], nt * me.np);
            if (me.np > 1) me.p0 = atomicAdd(&pslot_cur, nt * me.np);
        }
        grp[tid] = me;
        __syncthreads();
        for (int i = warp; i < min(1024, n_groups - g0); i += 32) {
            const SimGroup q = grp[i];
            if (q.cnt == 0) continue;
            const int nt = (q.cnt + kTcTile - 1) / kTcTile, nb = key_blocks(q.len);
            for (int e = lane; e < nt * q.np; e += 32) {
                const int t = e / q.np, part = e - t * q.np, n = min(kTcTile, q.cnt - t * kTcTile);
                const int64_t pos0 = (int64_t)q.start + (int64_t)t * kTcTile;
                const int b0 = nb * part / q.np, b1 = nb * (part + 1) / q.np;
                if (q.j0 + e < job_cap) {   // (it is for a launch within the context's limits, sim_prepare)
                    const int j = place_of(q.j0 + e);
                    jobs[j] = JobDev{q.slot, n, pos0, q.np == 1 ? q.len : min(q.len - b0 * 128, (b1 - b0) * 128), q.key0 + b0 * 128, part, q.np,
                                            q.p0 + t * q.np, q.len};
                    if (part == 0 && q.np > 1) joins[atomicAdd(&join_cur, 1)] = j;
                }
            }
        }
        __syncthreads();
    }
    if (tid == 0) n_out[1] = join_cur;
}

struct SimPlan {
    int n_groups_max = 0;
    size_t tile_cap = 0, cap = 0;
    int32_t *grp_cnt = nullptr, *grp_start = nullptr, *ids_sorted = nullptr, *out_index = nullptr, *n_jobs_dev = nullptr;   // [2]: jobs, split tiles
    int2 *where = nullptr;       // [cap] group and rank of every candidate
    JobDev *jobs = nullptr;      // [tile_cap + kSplitSlots]
    int32_t *joins = nullptr;    // [kSplitSlots] first pieces of the split tiles
};

SimPlan *plan_of(const aif_ctx *ctx) { return reinterpret_cast<SimPlan *>(ctx->sim_plan); }

}  // namespace

// rows of a slot's grouped sequence: every sub-sequence rounded up to 128 rows
size_t sim_grouped_rows(int L_max, int n_categories) { return ((size_t)L_max + 127) / 128 * 128 + (size_t)n_categories * 128; }

cudaError_t sim_prepare(aif_ctx *ctx)
{
    const aif_config &c = ctx->cfg;
    SimPlan *pl = new SimPlan();
    ctx->sim_plan = pl;
    pl->n_groups_max = c.max_user_states * c.n_categories;
    pl->cap = (size_t)c.max_batch_candidates;
    // a group of n candidates is ceil(n / 128) tiles: at most candidates / 128 tiles plus one per non-empty group
    const size_t groups = (size_t)pl->n_groups_max < pl->cap ? (size_t)pl->n_groups_max : pl->cap;
    pl->tile_cap = pl->cap / kTcTile + groups + 1;
    auto alloc = [&](void **p, size_t bytes) -> cudaError_t {
        bytes = (bytes + 255) / 256 * 256;
        cudaError_t e = cudaMalloc(p, bytes);
        if (e != cudaSuccess) return e;
        ctx->allocations.push_back(*p);
        ctx->device_bytes += (int64_t)bytes;
        return cudaMemset(*p, 0, bytes);
    };
    cudaError_t e;
    if ((e = alloc((void **)&pl->grp_cnt, (size_t)pl->n_groups_max * 4)) != cudaSuccess) return e;
    if ((e = alloc((void **)&pl->grp_start, (size_t)pl->n_groups_max * 4)) != cudaSuccess) return e;
    if ((e = alloc((void **)&pl->ids_sorted, (pl->cap + kTcTile) * 4)) != cudaSuccess) return e;
    if ((e = alloc((void **)&pl->out_index, (pl->cap + kTcTile) * 4)) != cudaSuccess) return e;
    if ((e = alloc((void **)&pl->where, pl->cap * sizeof(int2))) != cudaSuccess) return e;
    if ((e = alloc((void **)&pl->n_jobs_dev, 256)) != cudaSuccess) return e;
    if ((e = alloc((void **)&pl->jobs, (pl->tile_cap + kSplitSlots) * sizeof(JobDev))) != cudaSuccess) return e;
    if ((e = alloc((void **)&pl->joins, kSplitSlots * 4)) != cudaSuccess) return e;
    return cudaSuccess;
}

void sim_destroy(aif_ctx *ctx)
{
    delete plan_of(ctx);
    ctx->sim_plan = nullptr;
}

cudaError_t sim_group_sequence(const aif_ctx *ctx, HostSlot &hs, const int32_t *seq_cat, int L, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    const int nb = (L + kCatBlock - 1) / kCatBlock;
    cudaError_t e;
    k_cat_hist<<<nb, kCatBlock, (size_t)c.n_categories * 4, st>>>(seq_cat, L, c.n_categories, hs.cat_hist, ctx->status);
    k_cat_scan<<<1, kCatBlock, 0, st>>>(nb, c.n_categories, hs.cat_hist, const_cast<int32_t *>(hs.dev.cat_off),
                                        const_cast<int32_t *>(hs.dev.cat_len));
    k_cat_place<<<nb, kCatBlock, 0, st>>>(seq_cat, L, c.n_categories, hs.cat_hist, hs.dev.cat_off, hs.cat_map);
    count_launch(3);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // zero rows everywhere (the padding of every sub-sequence), then the items at their places
    const size_t row_bytes = (size_t)c.d * ctx->el;
    if ((e = cudaMemsetAsync(const_cast<void *>(hs.dev.Sg), 0, ctx->grouped_rows * row_bytes, st)) != cudaSuccess) return e;
    const int64_t vecs = (int64_t)L * (int64_t)(row_bytes / 16);
    k_group_rows<<<(int)((vecs + 255) / 256 < 1184 ? (vecs + 255) / 256 : 1184), 256, 0, st>>>(
        (const uint4 *)hs.dev.S, hs.cat_map, L, (int)(row_bytes / 16), (uint4 *)const_cast<void *>(hs.dev.Sg));
    count_launch();
    if (hs.dev.sigEg) {
        if ((e = cudaMemsetAsync(const_cast<uint8_t *>(hs.dev.sigEg), 0, ctx->grouped_rows * (size_t)c.lsh_bits, st)) != cudaSuccess) return e;
        const int64_t v2 = (int64_t)L * (c.lsh_bits / 16);
        k_group_rows<<<(int)((v2 + 255) / 256 < 1184 ? (v2 + 255) / 256 : 1184), 256, 0, st>>>(
            (const uint4 *)hs.dev.sigE, hs.cat_map, L, c.lsh_bits / 16, (uint4 *)const_cast<uint8_t *>(hs.dev.sigEg));
        count_launch();
    }
    return cudaGetLastError();
}

cudaError_t sim_group_candidates(const aif_ctx *ctx, ScoreLaunch &sl, SimPlace &place, TileDev *row_tiles, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    SimPlan *pl = plan_of(ctx);
    const int n_groups = sl.n_req * c.n_categories;
    const int grid = (int)((sl.total + 255) / 256 < 1184 ? (sl.total + 255) / 256 : 1184);
    cudaError_t e = launch_pdl(k_sim_count, dim3(grid), dim3(256), 0, st, sl, c.M, c.n_categories, c.bucket_mode, pl->grp_cnt, pl->where,
                               c.mini_batch, row_tiles);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_sim_tiles, dim3(1), dim3(1024), 0, st, sl, n_groups, c.n_categories, pl->grp_cnt, pl->grp_start, pl->jobs,
                   (int)pl->tile_cap + kSplitSlots, pl->joins, pl->n_jobs_dev);
    if (e != cudaSuccess) return e;
    count_launch(2);
    place = SimPlace{pl->where, pl->grp_start, pl->ids_sorted, pl->out_index};
    const int64_t groups = (int64_t)n_groups < sl.total ? (int64_t)n_groups : sl.total;
    sl.n_tiles = (int32_t)(sl.total / kTcTile + groups + 1 < (int64_t)pl->tile_cap ? sl.total / kTcTile + groups + 1 : (int64_t)pl->tile_cap);
    sl.joins = pl->joins, sl.jobs = pl->jobs, sl.n_jobs_dev = pl->n_jobs_dev, sl.n_jobs = sl.n_tiles + (sl.split.slots >= kSplitSlots ? kSplitSlots : 0);
    sl.out_index = pl->out_index;
    sl.grouped = 1;
    return cudaSuccess;
}

}  // namespace aif
