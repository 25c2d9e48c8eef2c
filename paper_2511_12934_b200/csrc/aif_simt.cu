// CUDA-core kernels of libaif: table refresh / gather and the general scoring kernel (any storage type, all
// interaction blocks, fp32 arithmetic).  The user-side network lives in aif_user.cu, the tensor-core kernels in aif_tc*.cu.
#include "aif_internal.h"
#include "aif_device.cuh"
#include "aif_tc_ptx.cuh"

namespace aif {

std::atomic<uint64_t> g_launches{0};

// ------------------------------------------------------------------------------------------------
// item table: scatter (nearline refresh) and gather
// ------------------------------------------------------------------------------------------------
// Rows of a sidecar (BEA weights, signatures) of the `rows` table rows a warp is at, in units of V: lane r of the warp holds
// row r's id in `my` (-1: outside the table).  SCATTER: src rows r0, r0 + 1, ... go to dst rows ids; else the other way round,
// with zeros for a bad id.
template <typename V, bool SCATTER>
__device__ __forceinline__ void move_side_units(const V *__restrict__ src, V *__restrict__ dst, int w, int rows, int64_t r0, int64_t n, int my)
{
    const int lane = threadIdx.x & 31;
    for (int b = 0; b < rows * w; b += 32) {
        const int i = b + lane, r = w == 1 ? i : i / w, c = i - r * w;
        const int id = __shfl_sync(0xffffffffu, my, r & 31);
        if (r >= rows || r0 + r >= n) continue;
        if (SCATTER) {
            if (id >= 0) dst[(int64_t)id * w + c] = src[(r0 + r) * w + c];
        } else
            dst[(r0 + r) * w + c] = id >= 0 ? src[(int64_t)id * w + c] : V{};
    }
}

struct SideRows {
    const void *src;
    void *dst;
    int32_t bytes;   // of a row; 0: no such sidecar in this launch
    int32_t unit;    // bytes moved at a time: the largest of 16, 8, 4, 2, 1 that divides the row and both addresses
};

template <bool SCATTER>
__device__ __forceinline__ void move_side(const SideRows &s, int rows, int64_t r0, int64_t n, int my)
{
    if (s.bytes == 0) return;
    if (s.unit == 16) move_side_units<uint4, SCATTER>((const uint4 *)s.src, (uint4 *)s.dst, s.bytes / 16, rows, r0, n, my);
    else if (s.unit == 8) move_side_units<uint2, SCATTER>((const uint2 *)s.src, (uint2 *)s.dst, s.bytes / 8, rows, r0, n, my);
    else if (s.unit == 4) move_side_units<uint32_t, SCATTER>((const uint32_t *)s.src, (uint32_t *)s.dst, s.bytes / 4, rows, r0, n, my);
    else if (s.unit == 2) move_side_units<uint16_t, SCATTER>((const uint16_t *)s.src, (uint16_t *)s.dst, s.bytes / 2, rows, r0, n, my);
    else move_side_units<uint8_t, SCATTER>((const uint8_t *)s.src, (uint8_t *)s.dst, s.bytes, rows, r0, n, my);
}

static SideRows side_rows(const void *src, void *dst, size_t bytes)
{
    SideRows s{src, dst, (int32_t)bytes, 16};
    while (s.unit > 1 && (bytes | (uintptr_t)src | (uintptr_t)dst) % s.unit) s.unit >>= 1;
    return s;
}

__device__ __forceinline__ float sum_squares(const uint4 &v, float)
{
    const float a = __uint_as_float(v.x), b = __uint_as_float(v.y), c = __uint_as_float(v.z), d = __uint_as_float(v.w);
    return fmaf(a, a, fmaf(b, b, fmaf(c, c, d * d)));
}
__device__ __forceinline__ float sum_squares(const uint4 &v, __nv_bfloat16)
{
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(h[i]);
        acc = fmaf(f.x, f.x, fmaf(f.y, f.y, acc));
    }
    return acc;
}

// Nearline refresh in one pass: table[ids[i]] = rows[i] with both sidecars, and the table's norm bound raised to the largest
// Euclidean norm of the rows written (norm_max may be null: bound already known).  Bound by memory traffic, each row read
// once and written once: the rows in flight are in registers when the norm is formed, so no second pass reads the table.
// A warp takes 8 x (32 / G) rows per step, G lanes of 16 bytes per row: one coalesced load brings their ids, handed round by
// shuffles, and every lane has eight independent loads in flight.  Norms are non-negative, so their bit patterns order like
// integers; a NaN row yields a pattern above every finite one and stays.
// Measured, 10^5 rows of 256 bytes with two 16-byte sidecars: 13 us (4.5 TB/s, the ids scatter the writes); as three scatter
// launches, a 64-bit division per vector, and a norm pass over the table 45 us from first to last.
template <typename T, int G>
__global__ void __launch_bounds__(256) k_refresh_rows(uint4 *__restrict__ table, const uint4 *__restrict__ rows, const int32_t *__restrict__ ids,
                                                      int64_t n, int vpr, int64_t M, SideRows bea, SideRows sig, float *norm_max,
                                                      uint32_t *status)
{
    grid_dep_launch();
    grid_dep_wait();
    constexpr int RPI = 32 / G, RPS = 8 * RPI;
    const int lane = threadIdx.x & 31, sub = lane / G, c = lane % G;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int best = 0;
    for (int64_t r0 = warp * RPS; r0 < n; r0 += n_warps * RPS) {
        // the ids and the first vectors of all rows are requested together: the ids are needed only for the stores
        int64_t dst_row = -1;
        const bool has_id = lane < RPS && r0 + lane < n;
        if (has_id) dst_row = ids ? (int64_t)ids[r0 + lane] : r0 + lane;
        float ss[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) ss[u] = 0.f;
        int my = -1;
        for (int c0 = c; c0 - c < vpr; c0 += G) {
            uint4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int64_t r = r0 + u * RPI + sub;
                v[u] = r < n && c0 < vpr ? __ldcs(rows + r * vpr + c0) : make_uint4(0, 0, 0, 0);
            }
            my = dst_row >= 0 && dst_row < M ? (int)dst_row : -1;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int dst = __shfl_sync(0xffffffffu, my, u * RPI + sub);
                if (dst >= 0 && c0 < vpr) {
                    table[(int64_t)dst * vpr + c0] = v[u];
                    ss[u] += sum_squares(v[u], T());
                }
            }
        }
        if (has_id && my < 0) atomicOr(status, AIF_STATUS_BAD_ID);
        if (norm_max) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) ss[u] += __shfl_xor_sync(0xffffffffu, ss[u], o);
                best = max(best, __float_as_int(sqrtf(ss[u])) & 0x7fffffff);
            }
        }
        move_side<true>(bea, RPS, r0, n, my);
        move_side<true>(sig, RPS, r0, n, my);
    }
    if (norm_max) {
        best = __reduce_max_sync(0xffffffffu, best);
        if (lane == 0 && best > 0) atomicMax(reinterpret_cast<int *>(norm_max), best);
    }
}

// rows_out[i] = table[ids[i]]; 16 bytes per thread and four independent rows in flight per thread.
__global__ void __launch_bounds__(256) k_gather_rows(const uint4 *__restrict__ table, const int32_t *__restrict__ ids,
                                                     int64_t n, int vec_per_row, int64_t M, uint4 *__restrict__ out,
                                                     uint32_t *status)
{
    const int64_t total = n * vec_per_row;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i < total; i += 4 * stride) {
        uint4 v[4];
        bool ok[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t ii = i + u * stride;
            ok[u] = false;
            v[u] = make_uint4(0, 0, 0, 0);
            if (ii < total) {
                const int64_t r = ii / vec_per_row;
                const int c = (int)(ii - r * vec_per_row);
                const int64_t src = ids[r];
                ok[u] = true;
                if (src >= 0 && src < M) v[u] = __ldg(table + src * vec_per_row + c);
                else if (c == 0) atomicOr(status, AIF_STATUS_BAD_ID);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (ok[u]) out[i + u * stride] = v[u];
    }
}

// Copies candidate ids from page-locked host memory that is mapped into the device's address space.
__global__ void __launch_bounds__(256) k_stage_ids(const int32_t *__restrict__ src, int32_t *__restrict__ dst, int64_t n)
{
    grid_dep_launch();
    grid_dep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) dst[i] = src[i];
}

cudaError_t launch_stage_ids(const int32_t *mapped_src, int32_t *dst, int64_t n, cudaStream_t st)
{
    const int grid = (int)((n + 255) / 256 < 592 ? (n + 255) / 256 : 592);
    const cudaError_t e = launch_pdl(k_stage_ids, dim3(grid), dim3(256), 0, st, mapped_src, dst, n);
    count_launch();
    return e;
}

static int grid_for(int64_t items, int per_block, int cap)
{
    int64_t g = (items + per_block - 1) / per_block;
    if (g < 1) g = 1;
    return (int)(g > cap ? cap : g);
}

template <typename T>
static cudaError_t refresh_typed(const aif_ctx *ctx, const int32_t *ids, int64_t n, const void *rows, const SideRows &bea, const SideRows &sig,
                                 float *norm_max, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    const int vpr = (int)((size_t)c.d * ctx->el / 16);   // d is a multiple of 32: whole 16-byte vectors
    const int G = vpr <= 8 ? 8 : vpr <= 16 ? 16 : 32, rps = 8 * (32 / G);
    const int grid = grid_for((n + rps - 1) / rps, 8, 148 * 8);
    auto go = [&](auto kernel) {
        return launch_pdl(kernel, dim3(grid), dim3(256), 0, st, (uint4 *)ctx->E, (const uint4 *)rows, ids, n, vpr, c.M, bea, sig, norm_max, ctx->status);
    };
    const cudaError_t e = G == 8 ? go(k_refresh_rows<T, 8>) : G == 16 ? go(k_refresh_rows<T, 16>) : go(k_refresh_rows<T, 32>);
    count_launch();
    return e;
}

cudaError_t launch_refresh_rows(const aif_ctx *ctx, const int32_t *ids, int64_t n, const void *rows, const void *bea_w, const uint8_t *sig,
                                float *norm_max, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    SideRows sb{}, ss{};
    if (ctx->bea_w) sb = side_rows(bea_w, ctx->bea_w, (size_t)c.n_bridge * ctx->el);
    if (ctx->sig) ss = side_rows(sig, ctx->sig, (size_t)c.lsh_bits / 8);
    return c.dtype == AIF_F32 ? refresh_typed<float>(ctx, ids, n, rows, sb, ss, norm_max, st)
                              : refresh_typed<__nv_bfloat16>(ctx, ids, n, rows, sb, ss, norm_max, st);
}

// The same for rows of VPR 16-byte vectors with VPR a divisor of 32 (128 to 512 bytes: every benchmark shape).  A warp
// takes 8 x (32 / VPR) consecutive output rows per step: their ids arrive with one coalesced load and are handed round by
// shuffles, every lane then has eight independent 16-byte loads in flight, each instruction covering whole rows, and no
// division or second dependent load stands between a lane and its data.
template <int VPR>
__global__ void __launch_bounds__(256) k_gather_rows_w(const uint4 *__restrict__ table, const int32_t *__restrict__ ids, int64_t n, int64_t M,
                                                       uint4 *__restrict__ out, uint32_t *status)
{
    grid_dep_launch();
    grid_dep_wait();
    constexpr int RPI = 32 / VPR, RPS = 8 * RPI;   // rows per instruction, rows per step of a warp
    const int lane = threadIdx.x & 31, sub = lane / VPR, c = lane % VPR;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r0 = warp * RPS; r0 < n; r0 += n_warps * RPS) {
        int my = -1;
        if (lane < RPS && r0 + lane < n) {
            my = ids[r0 + lane];
            if (my < 0 || (int64_t)my >= M) {
                my = -1;
                atomicOr(status, AIF_STATUS_BAD_ID);
            }
        }
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int src = __shfl_sync(0xffffffffu, my, u * RPI + sub);
            v[u] = src >= 0 ? __ldg(table + (int64_t)src * VPR + c) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t r = r0 + u * RPI + sub;
            if (r < n) __stcs(out + r * VPR + c, v[u]);
        }
    }
}

cudaError_t launch_gather_rows(const aif_ctx *ctx, const int32_t *ids, int64_t n, void *out, cudaStream_t st)
{
    const int vpr = (int)((size_t)ctx->cfg.d * ctx->el / 16);
    if (vpr == 8 || vpr == 16 || vpr == 32) {
        const int rps = 8 * (32 / vpr);
        const int64_t warps = (n + rps - 1) / rps;
        const int grid = (int)((warps + 7) / 8 < 148 * 16 ? (warps + 7) / 8 : 148 * 16);
        auto go = [&](auto kernel) {
            return launch_pdl(kernel, dim3(grid), dim3(256), 0, st, (const uint4 *)ctx->E, ids, n, ctx->cfg.M, (uint4 *)out, ctx->status);
        };
        const cudaError_t e = vpr == 8 ? go(k_gather_rows_w<8>) : vpr == 16 ? go(k_gather_rows_w<16>) : go(k_gather_rows_w<32>);
        count_launch();
        return e;
    }
    const int64_t total = n * vpr;
    const int grid = grid_for((total + 3) / 4, 256, 148 * 16);
    k_gather_rows<<<grid, 256, 0, st>>>((const uint4 *)ctx->E, ids, n, vpr, ctx->cfg.M, (uint4 *)out, ctx->status);
    count_launch();
    return cudaGetLastError();
}

// The sidecars of rows ids[0..n): a warp takes 32 rows per step, their ids with one coalesced load, both sidecars in the same
// launch (as two launches of one 4-byte word per thread: 7.9 + 7.2 us for 2.6e5 rows of 16 + 16 bytes).
__global__ void __launch_bounds__(256) k_gather_sidecars(const int32_t *__restrict__ ids, int64_t n, int64_t M, SideRows bea, SideRows sig,
                                                         uint32_t *status)
{
    grid_dep_launch();
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r0 = warp * 32; r0 < n; r0 += n_warps * 32) {
        int my = -1;
        if (r0 + lane < n) {
            my = ids[r0 + lane];
            if (my < 0 || (int64_t)my >= M) {
                my = -1;
                atomicOr(status, AIF_STATUS_BAD_ID);
            }
        }
        move_side<false>(bea, 32, r0, n, my);
        move_side<false>(sig, 32, r0, n, my);
    }
}

cudaError_t launch_gather_sidecars(const aif_ctx *ctx, const int32_t *ids, int64_t n, void *bea_w_out, uint8_t *sig_out, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    SideRows sb{}, ss{};
    if (bea_w_out) sb = side_rows(ctx->bea_w, bea_w_out, (size_t)c.n_bridge * ctx->el);
    if (sig_out) ss = side_rows(ctx->sig, sig_out, (size_t)c.lsh_bits / 8);
    const cudaError_t e = launch_pdl(k_gather_sidecars, dim3(grid_for((n + 31) / 32, 8, 148 * 16)), dim3(256), 0, st, ids, n, c.M, sb, ss, ctx->status);
    count_launch();
    return e;
}

template <typename T>
__global__ void k_transpose(const T *__restrict__ in, T *__restrict__ out, int rows, int cols)
{
    __shared__ T tile[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int y = by + r, x = bx + threadIdx.x;
        if (y < rows && x < cols) tile[r][threadIdx.x] = in[(size_t)y * cols + x];
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int x = bx + r, y = by + threadIdx.x;
        if (y < rows && x < cols) out[(size_t)x * rows + y] = tile[threadIdx.x][r];
    }
}

// out [cols x rows] = in [rows x cols]^T
cudaError_t launch_transpose(const void *in, void *out, int rows, int cols, size_t el, cudaStream_t st)
{
    dim3 grid((cols + 31) / 32, (rows + 31) / 32), block(32, 8);
    if (el == 4) k_transpose<float><<<grid, block, 0, st>>>((const float *)in, (float *)out, rows, cols);
    else k_transpose<uint16_t><<<grid, block, 0, st>>>((const uint16_t *)in, (uint16_t *)out, rows, cols);
    count_launch();
    return cudaGetLastError();
}

int simt_tiles_for(const aif_ctx *ctx, int n) { return tiles_of(n, kSimtTile, ctx->cfg.mini_batch); }

// ------------------------------------------------------------------------------------------------
// general scoring kernel: one block = one tile of kSimtTile candidates, one warp per candidate for the
// interaction blocks, then all threads for the MLP with the decomposed first layer.
// ------------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kSimtThreads) k_score_simt(ModelDev md, ScoreLaunch sl, int max_h)
{
    constexpr int TM = kSimtTile;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *xs = reinterpret_cast<float *>(smem_raw);        // [k1][TM]   candidate-dependent input, transposed
    float *ha = xs + (size_t)md.k1 * TM;                     // [max_h][TM]
    float *hb = ha + (size_t)max_h * TM;                     // [max_h][TM]
    float *qv = hb + (size_t)max_h * TM;                     // [TM][d]    item vectors as fp32 rows (queries)
    uint32_t *sigq = reinterpret_cast<uint32_t *>(qv + (size_t)TM * md.d);   // [TM][8]
    int *tiers = reinterpret_cast<int *>(sigq + TM * 8);     // [TM][16]
    int *bkt = tiers + TM * 16;                              // [TM][F]
    int *id_s = bkt + TM * md.F;                             // [TM]

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const ReqDev rq = find_request(sl, blockIdx.x);
    int start, cnt;
    tile_range(blockIdx.x - rq.tile_begin, rq.n, TM, md.mini_batch, start, cnt);
    const SlotDev slot = sl.slots[rq.slot];
    const int32_t *ids = sl.ids + rq.off + start;
    float *logits = sl.logits + rq.off + start;
    const int d = md.d, dq = d >> 5;

    if (tid < TM) {
        int id = -1;
        if (tid < cnt) {
            id = ids[tid];
            if (id < 0 || (int64_t)id >= md.M) {
                id = -1;
                atomicOr(sl.status, AIF_STATUS_BAD_ID);
            }
        }
        id_s[tid] = id;
    }
    for (int i = tid; i < md.k1 * TM; i += kSimtThreads) xs[i] = 0.f;
    for (int i = tid; i < TM * 16; i += kSimtThreads) tiers[i] = 0;
    __syncthreads();

    // ---- stage A: interaction blocks, warp c <-> candidate c
    {
        const int c = warp;
        const int id = id_s[c];
        if (id >= 0) {
            const T *e = reinterpret_cast<const T *>(md.E) + (size_t)id * d;
            int col = 0;
            for (int k = lane; k < d; k += 32) {
                const float v = to_f(e[k]);
                qv[c * d + k] = v;
                xs[(col + k) * TM + c] = v;
            }
            col += d;
            const bool do_att = md.blocks & AIF_BLK_ATT, do_din = md.blocks & AIF_BLK_LSH_DIN,
                       do_tier = md.blocks & AIF_BLK_SIMTIER, do_lsh = do_din || do_tier;
            if (do_lsh && lane < (md.lsh_bits >> 5))
                sigq[c * 8 + lane] = reinterpret_cast<const uint32_t *>(md.sig + (size_t)id * (md.lsh_bits >> 3))[lane];
            if (md.blocks & AIF_BLK_CROSS)
                for (int f = lane; f < md.F; f += 32) bkt[c * md.F + f] = bucket_of(id, f, md.B, md.bucket_mode);
            __syncwarp();
            float att[8], din[8];
            if (do_att || do_lsh)
                warp_interact<T>(qv + c * d, reinterpret_cast<const T *>(slot.S), slot.L, d, rsqrtf((float)d), do_att,
                                 do_lsh, do_tier, sigq + c * 8, slot.sigS, md.lsh_bits, md.n_tiers, tiers + c * 16, att,
                                 din);
            if (do_att) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < dq) xs[(col + lane + 32 * q) * TM + c] = att[q];
                col += d;
            }
            if (md.blocks & AIF_BLK_CROSS) {
                const T *Tt = reinterpret_cast<const T *>(slot.T);
                const int fdc = md.F * md.dc;
                for (int i = lane; i < fdc; i += 32) {
                    const int f = i / md.dc, k = i - f * md.dc;
                    xs[(col + i) * TM + c] = to_f(Tt[((size_t)f * md.B + bkt[c * md.F + f]) * md.dc + k]);
                }
                col += fdc;
            }
            if (md.blocks & AIF_BLK_BEA) {
                const T *wh = reinterpret_cast<const T *>(md.bea_w) + (size_t)id * md.n_bridge;
                const T *V = reinterpret_cast<const T *>(slot.V);
                for (int k = lane; k < d; k += 32) {
                    float acc = 0.f;
                    for (int b = 0; b < md.n_bridge; ++b) acc = fmaf(to_f(wh[b]), to_f(V[(size_t)b * d + k]), acc);
                    xs[(col + k) * TM + c] = acc;
                }
                col += d;
            }
            if (do_din) {
                const float nrm = md.lsh_din_norm == AIF_NORM_MEAN ? 1.0f / (float)slot.L : 1.0f;
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < dq) xs[(col + lane + 32 * q) * TM + c] = din[q] * nrm;
                col += d;
            }
            if (do_tier) {
                __syncwarp();
                const float nrm = md.simtier_norm == AIF_NORM_MEAN ? 1.0f / (float)slot.L : 1.0f;
                if (lane < md.n_tiers) xs[(col + lane) * TM + c] = (float)tiers[c * 16 + lane] * nrm;
            }
        }
    }
    __syncthreads();

    // ---- stage B: MLP.  First layer = cached user partial + candidate-dependent columns.
    const float *in_act = xs;
    float *out_act = ha;
    int in_w = md.k1;
    for (int layer = 0; layer < md.n_hidden; ++layer) {
        const int H = md.hidden[layer];
        const T *W = reinterpret_cast<const T *>(md.Wt[layer]) + (layer == 0 ? (size_t)d * H : 0);
        const float *bias = layer == 0 ? slot.p_u : md.b[layer];
        for (int j = tid; j < H; j += kSimtThreads) {
            float acc[TM];
            const float b0 = bias[j];
#pragma unroll
            for (int c = 0; c < TM; ++c) acc[c] = b0;
            // weights in batches of 32 independent loads (the accumulation order over k stays sequential): after an L2
            // flush every weight comes from HBM, and one load per iteration would expose that latency 32 times as often
            auto step = [&](int k, float w) {
                const float4 a = *reinterpret_cast<const float4 *>(in_act + k * TM);
                const float4 b = *reinterpret_cast<const float4 *>(in_act + k * TM + 4);
                acc[0] = fmaf(w, a.x, acc[0]);
                acc[1] = fmaf(w, a.y, acc[1]);
                acc[2] = fmaf(w, a.z, acc[2]);
                acc[3] = fmaf(w, a.w, acc[3]);
                acc[4] = fmaf(w, b.x, acc[4]);
                acc[5] = fmaf(w, b.y, acc[5]);
                acc[6] = fmaf(w, b.z, acc[6]);
                acc[7] = fmaf(w, b.w, acc[7]);
            };
            int k = 0;
            for (; k + 32 <= in_w; k += 32) {
                float w[32];
#pragma unroll
                for (int u = 0; u < 32; ++u) w[u] = to_f(W[(size_t)(k + u) * H + j]);
#pragma unroll
                for (int u = 0; u < 32; ++u) step(k + u, w[u]);
            }
            for (; k < in_w; ++k) step(k, to_f(W[(size_t)k * H + j]));
#pragma unroll
            for (int c = 0; c < TM; ++c) out_act[j * TM + c] = fmaxf(acc[c], 0.f);
        }
        __syncthreads();
        in_act = out_act;
        out_act = (out_act == ha) ? hb : ha;
        in_w = H;
    }
    // ---- output layer: warp c reduces candidate c in a fixed order
    {
        const int c = warp;
        if (c < cnt) {
            const T *wo = reinterpret_cast<const T *>(md.w_out);
            float acc = 0.f;
            for (int j = lane; j < in_w; j += 32) acc = fmaf(to_f(wo[j]), in_act[j * TM + c], acc);
            acc = warp_sum(acc);
            if (lane == 0) {
                float logit = acc + md.b_out[0];
                if (md.emit_sigmoid) logit = 1.0f / (1.0f + expf(-logit));
                logits[c] = id_s[c] >= 0 ? logit : __int_as_float(0x7fc00000);
            }
        }
    }
}

static size_t simt_smem_bytes(const aif_ctx *ctx, int &max_h)
{
    const aif_config &c = ctx->cfg;
    max_h = 0;
    for (int k = 0; k < c.n_hidden; ++k) max_h = c.hidden[k] > max_h ? c.hidden[k] : max_h;
    const int k1 = ctx->input_width - c.d;
    size_t fl = (size_t)(k1 + 2 * max_h + c.d) * kSimtTile;
    size_t ints = (size_t)kSimtTile * (8 + 16 + c.F + 1);
    return (fl + ints) * 4 + 16;
}

cudaError_t launch_score_simt(const aif_ctx *ctx, const ScoreLaunch &sl, cudaStream_t st)
{
    if (sl.n_tiles <= 0) return cudaSuccess;
    int max_h;
    const size_t smem = simt_smem_bytes(ctx, max_h);
    const ModelDev md = make_model(ctx);
    cudaError_t e;
    timing_begin(ctx, st);
    if (ctx->cfg.dtype == AIF_F32) {
        e = cudaFuncSetAttribute(k_score_simt<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_score_simt<float><<<sl.n_tiles, kSimtThreads, smem, st>>>(md, sl, max_h);
    } else {
        e = cudaFuncSetAttribute(k_score_simt<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_score_simt<__nv_bfloat16><<<sl.n_tiles, kSimtThreads, smem, st>>>(md, sl, max_h);
    }
    count_launch();
    timing_mark(ctx, "score_simt", st);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// norm bound over a set of rows
// ------------------------------------------------------------------------------------------------
// Largest Euclidean norm over a set of rows, one warp per row.  Norms are non-negative, so their bit patterns order like
// integers; a NaN row yields a pattern above every finite one and stays.
template <typename T>
__global__ void __launch_bounds__(256) k_row_norm_max(const T *__restrict__ rows, int64_t n, int d, float *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t w0 = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5), stride = (int64_t)gridDim.x * 8;
    int best = 0;
    for (int64_t i = w0; i < n; i += stride) {
        const T *row = rows + (size_t)i * d;
        float acc = 0.f;
        for (int c = lane; c < d; c += 32) {
            const float v = to_f(row[c]);
            acc = fmaf(v, v, acc);
        }
        acc = warp_sum(acc);
        best = max(best, __float_as_int(sqrtf(acc)) & 0x7fffffff);
    }
    if (lane == 0 && best > 0) atomicMax(reinterpret_cast<int *>(out), best);
}

cudaError_t launch_row_norm_max(const aif_ctx *ctx, const void *rows, int64_t n, float *out, cudaStream_t st)
{
    if (n <= 0 || !out) return cudaSuccess;
    const int64_t want = (n + 7) / 8;
    const int grid = (int)(want < 148 * 8 ? want : 148 * 8);
    if (ctx->cfg.dtype == AIF_F32) k_row_norm_max<float><<<grid, 256, 0, st>>>((const float *)rows, n, ctx->cfg.d, out);
    else k_row_norm_max<__nv_bfloat16><<<grid, 256, 0, st>>>((const __nv_bfloat16 *)rows, n, ctx->cfg.d, out);
    count_launch();
    return cudaGetLastError();
}

}  // namespace aif
