// CUDA-core kernels of libaif: table refresh / gather and the general scoring kernel (any storage type, all
// interaction blocks, fp32 arithmetic).  The user-side network lives in aif_user.cu, the tensor-core kernels in aif_tc*.cu.
#include <type_traits>

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

// Sidecar rows of one 16-byte unit (eight bf16 bridge weights, 128 signature bits): a lane moves its row's in one piece, so the loads of
// both sidecars go out with the others of a step instead of after its stores.
__device__ __forceinline__ bool one_unit(const SideRows &s) { return s.bytes == 16 && s.unit == 16; }

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
// SIDE: the table has sidecars.  Three blocks to an SM in either copy (3 x 10^5 rows and their gather: 48.4 us, with sidecars 62.4; with the 122
// registers that the compiler would take for rows alone 52.1; sidecars asked for behind the row stores 68.9).
template <typename T, int G, bool SIDE>
__global__ void __launch_bounds__(256, 3) k_refresh_rows(uint4 *__restrict__ table, const uint4 *__restrict__ rows, const int32_t *__restrict__ ids,
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
        const bool bea_one = SIDE && one_unit(bea), sig_one = SIDE && one_unit(sig);
        uint4 bea_v = make_uint4(0, 0, 0, 0), sig_v = bea_v;
        if (has_id && bea_one) bea_v = __ldcs(reinterpret_cast<const uint4 *>(bea.src) + r0 + lane);
        if (has_id && sig_one) sig_v = __ldcs(reinterpret_cast<const uint4 *>(sig.src) + r0 + lane);
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
        if (SIDE) {
            if (!bea_one) move_side<true>(bea, RPS, r0, n, my);
            else if (my >= 0) reinterpret_cast<uint4 *>(bea.dst)[my] = bea_v;
            if (!sig_one) move_side<true>(sig, RPS, r0, n, my);
            else if (my >= 0) reinterpret_cast<uint4 *>(sig.dst)[my] = sig_v;
        }
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
    auto pick = [&](auto side) {
        constexpr bool kSide = decltype(side)::value;
        return G == 8 ? go(k_refresh_rows<T, 8, kSide>) : G == 16 ? go(k_refresh_rows<T, 16, kSide>) : go(k_refresh_rows<T, 32, kSide>);
    };
    const cudaError_t e = bea.bytes || sig.bytes ? pick(std::true_type{}) : pick(std::false_type{});
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
        const bool bea_one = one_unit(bea), sig_one = one_unit(sig);
        uint4 bea_v = make_uint4(0, 0, 0, 0), sig_v = bea_v;
        if (my >= 0 && bea_one) bea_v = reinterpret_cast<const uint4 *>(bea.src)[my];
        if (my >= 0 && sig_one) sig_v = reinterpret_cast<const uint4 *>(sig.src)[my];
        if (!bea_one) move_side<false>(bea, 32, r0, n, my);
        else if (r0 + lane < n) __stcs(reinterpret_cast<uint4 *>(bea.dst) + r0 + lane, bea_v);
        if (!sig_one) move_side<false>(sig, 32, r0, n, my);
        else if (r0 + lane < n) __stcs(reinterpret_cast<uint4 *>(sig.dst) + r0 + lane, sig_v);
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
// General scoring kernel (fp32, and bf16 shapes the tensor-core kernels do not take): one block = one tile of kSimtTile
// candidates, a warp per candidate for the interaction blocks, then all of them for the MLP with the decomposed first layer.
// A request of 1000 candidates is 125 blocks, so what counts is the length of one block's dependent chain.  A block has
// 8 x (k1 H1 + H1 H2 + ..) multiply-adds to issue (6.1 k cycles for 256 -> 256 -> 128) and as many weight bytes to take in
// (393 KB at 59 bytes per clock: 6.7 k); everything else is kept short of that:
//   * key rows go through shared memory, 32 at a time, once per block; a lane scores one key from padded rows (conflict-free
//     16-byte reads).  Read from global memory by every warp, a whole row per lane and then once more key by key, 50 keys cost
//     more than the MLP.
//   * the weights come through a ring of 32 KB stages (bulk copies, requested by a warp of their own) from the kernel's first
//     moment on, across the layers; loaded by the threads that multiply, at most 32 KB were in flight and a layer waited for
//     every batch.
//   * shared memory returns 128 bytes per clock, broadcasts at full width: a lane's tile is 8 outputs x 8 candidates, 64 bytes per
//     64 multiply-adds and row (one output x 8 candidates, 36 bytes per 8: four times the multiply-adds' own time).  A warp takes
//     64 outputs, its lanes every fourth row of a stage, the next row's reads under this one's products; the four partial sums
//     meet in 48 shuffles, those of the warps that share 64 outputs in shared memory.
// Measured, 1000 candidates, 50 keys, d 64, fp32, from the call to the logits: 29.3 -> 16.8 us (the weight ring alone 22.9; 16 warps,
// two per candidate, at half the registers: 21.4, bound by instructions that were not products).  Now 17 of 31 k cycles are the
// MLP (10 in the products), 6 the attention, 5 the ids and rows.
// ------------------------------------------------------------------------------------------------
template <int DQ>
__device__ __forceinline__ float dot_shared(const float *row, const float *q)
{
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 32 * DQ; k += 4) {
        const float4 r = *reinterpret_cast<const float4 *>(row + k), w = *reinterpret_cast<const float4 *>(q + k);
        acc[0] = fmaf(r.x, w.x, acc[0]), acc[1] = fmaf(r.y, w.y, acc[1]), acc[2] = fmaf(r.z, w.z, acc[2]), acc[3] = fmaf(r.w, w.w, acc[3]);
    }
    return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}
template <int DQ>
__device__ __forceinline__ float dot_shared(const __nv_bfloat16 *row, const float *q)
{
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 32 * DQ; k += 8) {
        const uint4 r = *reinterpret_cast<const uint4 *>(row + k);
        const float4 a = *reinterpret_cast<const float4 *>(q + k), b = *reinterpret_cast<const float4 *>(q + k + 4);
        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&r);
        const float2 f0 = __bfloat1622float2(h[0]), f1 = __bfloat1622float2(h[1]), f2 = __bfloat1622float2(h[2]), f3 = __bfloat1622float2(h[3]);
        acc[0] = fmaf(f0.x, a.x, acc[0]), acc[1] = fmaf(f0.y, a.y, acc[1]), acc[2] = fmaf(f1.x, a.z, acc[2]), acc[3] = fmaf(f1.y, a.w, acc[3]);
        acc[0] = fmaf(f2.x, b.x, acc[0]), acc[1] = fmaf(f2.y, b.y, acc[1]), acc[2] = fmaf(f3.x, b.z, acc[2]), acc[3] = fmaf(f3.y, b.w, acc[3]);
    }
    return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}
__device__ __forceinline__ float4 load4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p)
{
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

constexpr int kSimtKeys = 32;            // keys of a chunk
constexpr int kSimtWarps = kSimtTile, kSimtThreads = 32 * kSimtWarps;   // a warp per candidate; one warp more requests the weights
constexpr int kSimtMaxStages = 4, kSimtStageBytes = 32768;
constexpr int kSimtRed = kSimtWarps * 64 * kSimtTile;   // floats: partial sums of the warps

// Shared memory of the kernel, in floats; the key chunks lie where the activations come later.
struct SimtLayout {
    int32_t max_h;
    int32_t region;      // of activations / key chunks
    int32_t key_bufs;    // chunk buffers, 2 or 1; 0: no room, keys are read from global memory
    int32_t stages;      // of the weight ring; 0: weights are read from global memory
    int32_t red, ps;     // partial sums (with the ring); probabilities and similarities of the key chunks
};

// Where the weights of the layers come from (launch_score_simt chooses): the ring, a block per SM and layers of at most kSimtRingH units;
// or global memory, a thread per output and 32 rows in flight per batch, with one block per SM and the registers for that
// (SIMT_DIRECT) or three blocks (SIMT_MANY): the same sums in the same order.
enum { SIMT_RING, SIMT_DIRECT, SIMT_MANY };
constexpr int kSimtRingH = 256, kSimtRingWeights = 65536;

// Rows of a layer of H units in one stage of the ring.
template <typename T>
__device__ __forceinline__ int simt_stage_rows(int H)
{
    return min(128, kSimtStageBytes / (H * (int)sizeof(T)));
}

// The weights of all layers, stage by stage, by one thread.
template <typename T>
__device__ __forceinline__ bool simt_weights(const ModelDev &md, unsigned char *ring, uint64_t *full, uint64_t *empty, int stages, volatile uint32_t *abort_flag)
{
    int s = 0, filled = 0;
    uint32_t ph = 1;
    for (int layer = 0; layer < md.n_hidden; ++layer) {
        const int H = md.hidden[layer], in_w = layer ? md.hidden[layer - 1] : md.k1;
        const T *W = reinterpret_cast<const T *>(md.Wt[layer]) + (layer == 0 ? (size_t)md.d * H : 0);
        const int stage_rows = simt_stage_rows<T>(H);
        for (int k0 = 0; k0 < in_w; k0 += stage_rows) {
            const uint32_t bar = smem_u32(full + s), bytes = (uint32_t)(min(stage_rows, in_w - k0) * H) * (uint32_t)sizeof(T);
            if (filled >= stages && !mbar_wait(smem_u32(empty + s), ph, abort_flag)) return false;
            mbar_expect_tx(bar, bytes);
            bulk_load(smem_u32(ring + s * kSimtStageBytes), W + (size_t)k0 * H, bytes, bar);
            ++filled;
            if (++s == stages) s = 0, ph ^= 1u;
        }
    }
    return true;
}

// The sequence blocks of one candidate by one warp (all warps in step: the chunks of keys are shared).
template <typename T, int DQ, typename Fetch>
__device__ __forceinline__ void simt_keys(const ModelDev &md, const uint8_t *sigS, int L, bool live, const float *q, const uint32_t *sigq,
                                          int *tiers, float *pp, float *pm, const unsigned char *keys, int n_bufs, float *xs_att,
                                          float *xs_din, Fetch fetch)
{
    constexpr int D = 32 * DQ, stride = D * (int)sizeof(T) + 16, TM = kSimtTile;
    const int lane = threadIdx.x & 31, n_chunks = (L + kSimtKeys - 1) / kSimtKeys, words = md.lsh_bits >> 5;
    const bool do_att = md.blocks & AIF_BLK_ATT, do_din = md.blocks & AIF_BLK_LSH_DIN, do_tier = md.blocks & AIF_BLK_SIMTIER;
    const float scale = rsqrtf((float)D), inv_bits = 1.0f / (float)md.lsh_bits;
    float att[DQ], din[DQ], m = -INFINITY, l = 0.f;
#pragma unroll
    for (int c = 0; c < DQ; ++c) att[c] = din[c] = 0.f;
    for (int ch = 0; ch < n_chunks; ++ch) {
        if (n_bufs == 2 && ch + 1 < n_chunks) cp_async_wait<1>();
        else cp_async_wait<0>();
        named_bar_sync(1, kSimtThreads);
        const unsigned char *buf = keys + (ch % n_bufs) * kSimtKeys * stride;
        if (live) {
            const int j = ch * kSimtKeys + lane;
            const bool valid = j < L;
            if (do_din || do_tier) {
                float simv = 0.f;
                if (valid) {
                    const uint32_t *sj = reinterpret_cast<const uint32_t *>(sigS + (size_t)j * (md.lsh_bits >> 3));
                    int diff = 0;
                    for (int w = 0; w < words; ++w) diff += __popc(sigq[w] ^ __ldg(sj + w));
                    const int matches = md.lsh_bits - diff;
                    simv = (float)matches * inv_bits;
                    if (do_tier) {
                        const int t = (matches * md.n_tiers) / md.lsh_bits;
                        atomicAdd(&tiers[t < md.n_tiers - 1 ? t : md.n_tiers - 1], 1);
                    }
                }
                pm[lane] = simv;
            }
            if (do_att) {
                const float s = valid ? dot_shared<DQ>(reinterpret_cast<const T *>(buf + lane * stride), q) * scale : -INFINITY;
                const float m_new = fmaxf(m, warp_max(s)), sc = expf(m - m_new), p = valid ? expf(s - m_new) : 0.f;
                pp[lane] = p;
                l = l * sc + warp_sum(p);
                m = m_new;
#pragma unroll
                for (int c = 0; c < DQ; ++c) att[c] *= sc;
            }
            __syncwarp();
            const int n = min(kSimtKeys, L - ch * kSimtKeys);   // up to three keys more: weight 0 times rows of zeros
            auto weigh = [&](const float *w, float (&acc)[DQ]) {
#pragma unroll 2
                for (int j0 = 0; j0 < n; j0 += 4) {
                    const float4 p4 = *reinterpret_cast<const float4 *>(w + j0);
                    const float pj[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const T *row = reinterpret_cast<const T *>(buf + (j0 + u) * stride) + lane;
#pragma unroll
                        for (int c = 0; c < DQ; ++c) acc[c] = fmaf(pj[u], to_f(row[32 * c]), acc[c]);
                    }
                }
            };
            if (do_att) weigh(pp, att);
            if (do_din) weigh(pm, din);
        }
        if (ch + n_bufs < n_chunks) {
            named_bar_sync(1, kSimtThreads);
            fetch(ch + n_bufs);
        }
    }
    if (!live) return;
    const float inv = 1.0f / l, nrm = md.lsh_din_norm == AIF_NORM_MEAN ? 1.0f / (float)L : 1.0f;
#pragma unroll
    for (int c = 0; c < DQ; ++c) {
        if (do_att) xs_att[(lane + 32 * c) * TM] = att[c] * inv;
        if (do_din) xs_din[(lane + 32 * c) * TM] = din[c] * nrm;
    }
}

template <typename T, int MODE>
__global__ void __launch_bounds__(MODE == SIMT_RING ? kSimtThreads + 32 : kSimtThreads, MODE == SIMT_MANY ? 3 : 1) k_score_simt(const __grid_constant__ ModelDev md, const __grid_constant__ ScoreLaunch sl, const SimtLayout lay)
{
    constexpr int TM = kSimtTile;
    constexpr bool RING = MODE == SIMT_RING;
    constexpr int kAll = RING ? kSimtThreads + 32 : kSimtThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *ring = smem_raw;
    float *xs = reinterpret_cast<float *>(smem_raw + (RING ? lay.stages * kSimtStageBytes : 0));   // [k1][TM] candidate-dependent input, transposed
    float *ha = xs + (size_t)md.k1 * TM;                     // [max_h][TM]
    float *hb = ha + (size_t)lay.max_h * TM;                 // [max_h][TM]
    unsigned char *keys = reinterpret_cast<unsigned char *>(ha);   // [key_bufs][kSimtKeys] rows of d elements and 16 bytes
    float *red = ha + lay.region;                            // [kSimtRed] partial sums of the layers
    float *qv = red + lay.red;                               // [TM][d]    item vectors as fp32 rows (queries)
    float *ps = qv + (size_t)TM * md.d;                      // [2][warp][kSimtKeys] probabilities, similarities
    uint32_t *sigq = reinterpret_cast<uint32_t *>(ps + lay.ps);   // [TM][8]
    int *tiers = reinterpret_cast<int *>(sigq + TM * 8);     // [TM][16]
    uint64_t *full = reinterpret_cast<uint64_t *>(tiers + TM * 16);   // (from here on with the ring only)
    uint64_t *empty = full + kSimtMaxStages;
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(empty + kSimtMaxStages);

    const int tid = threadIdx.x, lane = tid & 31, c = tid >> 5;   // candidate of this warp
    const int d = md.d;
    if (RING && tid == kSimtThreads) {
        for (int s = 0; s < kSimtMaxStages; ++s) mbar_init(smem_u32(full + s), 1), mbar_init(smem_u32(empty + s), kSimtWarps);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    grid_dep_launch();
    for (int i = tid; i < md.k1 * TM; i += kAll) xs[i] = 0.f;
    for (int i = tid; i < TM * 16; i += kAll) tiers[i] = 0;
    __syncthreads();   // xs is zero, the barriers exist
    if (RING && tid >= kSimtThreads) {
        // the weights are older than any launch this one may overlap: no wait for the previous kernel
        if (lane == 0 && !simt_weights<T>(md, ring, full, empty, lay.stages, abort_flag)) *abort_flag = 1u;
        return;
    }
    grid_dep_wait();
    const ReqDev rq = find_request(sl, blockIdx.x);
    int start, cnt;
    tile_range(blockIdx.x - rq.tile_begin, rq.n, TM, md.mini_batch, start, cnt);
    const SlotDev &slot = sl.slots[rq.slot];
    const int L = slot.L;
    const T *S = reinterpret_cast<const T *>(slot.S);
    int id = c < cnt ? sl.ids[rq.off + start + c] : -1;
    const float b_out = md.b_out[0];
    const bool do_att = md.blocks & AIF_BLK_ATT, do_din = md.blocks & AIF_BLK_LSH_DIN, do_tier = md.blocks & AIF_BLK_SIMTIER;
    const bool do_lsh = do_din || do_tier, chunked = lay.key_bufs && (do_att || do_lsh);
    const int row_bytes = d * (int)sizeof(T), stride = row_bytes + 16, vpr = row_bytes >> 4;
    auto fetch = [&](int ch) {   // keys beyond the sequence as zeros
        const uint32_t buf = smem_u32(keys + (ch % lay.key_bufs) * kSimtKeys * stride);
        for (int i = tid; i < kSimtKeys * vpr; i += kSimtThreads) {
            const int r = i / vpr, v = i - r * vpr, j = ch * kSimtKeys + r;
            cp_async16(buf + r * stride + v * 16, reinterpret_cast<const unsigned char *>(S) + (size_t)(j < L ? j : 0) * row_bytes + v * 16, j < L ? 16u : 0u);
        }
        cp_async_commit();
    };
    if (chunked) {
        fetch(0);
        if (lay.key_bufs == 2 && L > kSimtKeys) fetch(1);
    }
    if (id < 0 || (int64_t)id >= md.M) {
        id = -1;
        if (c < cnt && lane == 0) atomicOr(sl.status, AIF_STATUS_BAD_ID);
    }

    // ---- stage A: interaction blocks (a bad id keeps its zero columns but takes part in the barriers)
    {
        const int col_cross = d + (do_att ? d : 0), col_bea = col_cross + ((md.blocks & AIF_BLK_CROSS) ? md.F * md.dc : 0);
        const int col_din = col_bea + ((md.blocks & AIF_BLK_BEA) ? d : 0), col_tier = col_din + (do_din ? d : 0);
        if (id >= 0) {
            const T *e = reinterpret_cast<const T *>(md.E) + (size_t)id * d;
            for (int k0 = lane; k0 < d; k0 += 128) {
                float v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = k0 + 32 * u < d ? to_f(e[k0 + 32 * u]) : 0.f;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k0 + 32 * u < d) qv[c * d + k0 + 32 * u] = v[u], xs[(k0 + 32 * u) * TM + c] = v[u];
            }
            if (do_lsh && lane < (md.lsh_bits >> 5))
                sigq[c * 8 + lane] = reinterpret_cast<const uint32_t *>(md.sig + (size_t)id * (md.lsh_bits >> 3))[lane];
            if (md.blocks & AIF_BLK_BEA) {
                const T *wh = reinterpret_cast<const T *>(md.bea_w) + (size_t)id * md.n_bridge;
                const T *V = reinterpret_cast<const T *>(slot.V);
                for (int k = lane; k < d; k += 32) {
                    float acc = 0.f;
                    for (int b = 0; b < md.n_bridge; ++b) acc = fmaf(to_f(wh[b]), to_f(V[(size_t)b * d + k]), acc);
                    xs[(col_bea + k) * TM + c] = acc;
                }
            }
            if (md.blocks & AIF_BLK_CROSS) {
                const T *Tt = reinterpret_cast<const T *>(slot.T);
                // 32 fields at a time: a lane hashes one of them, once, the lanes that copy its elements get the bucket by shuffle
                // (a hash per element: 96 fields of 64, 1000 candidates, 326 us)
                for (int f0 = 0; f0 < md.F; f0 += 32) {
                    const int nf = min(32, md.F - f0), ne = nf * md.dc;
                    const int bucket = lane < nf ? bucket_of(id, f0 + lane, md.B, md.bucket_mode) : 0;
                    const T *Tf = Tt + (size_t)f0 * md.B * md.dc;
                    float *x = xs + (size_t)(col_cross + f0 * md.dc) * TM + c;
                    auto cell = [&](int i) {   // every lane of the warp, i < ne
                        const int f = i / md.dc;
                        return Tf + ((size_t)f * md.B + __shfl_sync(0xffffffffu, bucket, f)) * md.dc + (i - f * md.dc);
                    };
                    if (sizeof(T) == 4) {   // element by element straight to its place; the first layer waits for them
                        for (int i0 = 0; i0 < ne; i0 += 32) {
                            const T *src = cell(min(i0 + lane, ne - 1));
                            if (i0 + lane < ne) cp_async4(smem_u32(x + (i0 + lane) * TM), src);
                        }
                    } else
                        for (int i0 = lane; i0 - lane < ne; i0 += 128) {   // four independent reads per round
                            float v[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) v[u] = to_f(*cell(min(i0 + 32 * u, ne - 1)));
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (i0 + 32 * u < ne) x[(i0 + 32 * u) * TM] = v[u];
                        }
                }
            }
        }
        cp_async_commit();
        float *x_att = xs + d * TM + c, *x_din = xs + col_din * TM + c;
        if (chunked) {
            auto run = [&](auto dq) {
                simt_keys<T, decltype(dq)::value>(md, slot.sigS, L, id >= 0, qv + c * d, sigq + c * 8, tiers + c * 16, ps + c * kSimtKeys,
                                                  ps + (kSimtWarps + c) * kSimtKeys, keys, lay.key_bufs, x_att, x_din, fetch);
            };
            switch (d >> 5) {
                case 1: run(std::integral_constant<int, 1>{}); break;
                case 2: run(std::integral_constant<int, 2>{}); break;
                case 3: run(std::integral_constant<int, 3>{}); break;
                case 4: run(std::integral_constant<int, 4>{}); break;
                case 5: run(std::integral_constant<int, 5>{}); break;
                case 6: run(std::integral_constant<int, 6>{}); break;
                case 7: run(std::integral_constant<int, 7>{}); break;
                default: run(std::integral_constant<int, 8>{}); break;
            }
        } else if (id >= 0 && (do_att || do_lsh)) {
            __syncwarp();
            float att[8], din[8];
            warp_interact<T>(qv + c * d, S, L, d, rsqrtf((float)d), do_att, do_lsh, do_tier, sigq + c * 8, slot.sigS, md.lsh_bits, md.n_tiers,
                             tiers + c * 16, att, din);
            const float nrm = md.lsh_din_norm == AIF_NORM_MEAN ? 1.0f / (float)L : 1.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < (d >> 5)) {
                    if (do_att) x_att[(lane + 32 * q) * TM] = att[q];
                    if (do_din) x_din[(lane + 32 * q) * TM] = din[q] * nrm;
                }
        }
        if (do_tier && id >= 0) {
            __syncwarp();
            const float nrm = md.simtier_norm == AIF_NORM_MEAN ? 1.0f / (float)L : 1.0f;
            if (lane < md.n_tiers) xs[(col_tier + lane) * TM + c] = (float)tiers[c * 16 + lane] * nrm;
        }
    }

    // ---- stage B: MLP.  First layer = cached user partial + candidate-dependent columns.
    cp_async_wait_all();
    const float *in_act = xs;
    float *out_act = ha;
    int in_w = md.k1, s = 0;
    uint32_t ph = 0;
    bool ok = true, next = false;   // next: the stage after this one has been seen to be there
    const int ql = lane & 7, kp = lane >> 3;   // outputs 4 ql .. + 3 and 32 + 4 ql .. + 3 of the warp's 64; rows kp, kp + 4, ... of a stage
    for (int layer = 0; layer < md.n_hidden; ++layer) {
        const int H = md.hidden[layer];
        const float *bias = layer == 0 ? slot.p_u : md.b[layer];
        named_bar_sync(1, kSimtThreads);   // the layer's inputs are written
        if constexpr (!RING) {
            const T *W = reinterpret_cast<const T *>(md.Wt[layer]) + (layer == 0 ? (size_t)d * H : 0);
            for (int j = tid; j < H; j += kSimtThreads) {
                float acc[TM];
                const float b0 = bias[j];
#pragma unroll
                for (int cc = 0; cc < TM; ++cc) acc[cc] = b0;
                auto row = [&](int k, float w) {
                    const float4 a = *reinterpret_cast<const float4 *>(in_act + k * TM), b = *reinterpret_cast<const float4 *>(in_act + k * TM + 4);
                    acc[0] = fmaf(w, a.x, acc[0]), acc[1] = fmaf(w, a.y, acc[1]), acc[2] = fmaf(w, a.z, acc[2]), acc[3] = fmaf(w, a.w, acc[3]);
                    acc[4] = fmaf(w, b.x, acc[4]), acc[5] = fmaf(w, b.y, acc[5]), acc[6] = fmaf(w, b.z, acc[6]), acc[7] = fmaf(w, b.w, acc[7]);
                };
                int k = 0;
                for (; k + 32 <= in_w; k += 32) {
                    float w[32];
#pragma unroll
                    for (int u = 0; u < 32; ++u) w[u] = to_f(W[(size_t)(k + u) * H + j]);
#pragma unroll
                    for (int u = 0; u < 32; ++u) row(k + u, w[u]);
                }
                for (; k < in_w; ++k) row(k, to_f(W[(size_t)k * H + j]));
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *reinterpret_cast<float4 *>(out_act + (size_t)j * TM + 4 * h) =
                        make_float4(fmaxf(acc[4 * h], 0.f), fmaxf(acc[4 * h + 1], 0.f), fmaxf(acc[4 * h + 2], 0.f), fmaxf(acc[4 * h + 3], 0.f));
            }
        } else {
            const int stage_rows = simt_stage_rows<T>(H);
            const int groups = (H + 63) >> 6, splits = kSimtWarps / groups;   // groups of 64 outputs; warps per group
            const int grp = c % groups, part = c / groups;
            const bool busy = part < splits;
            uint64_t acc2[8][TM / 2];   // two candidates per register pair: half the instructions (f32x2)
#pragma unroll
            for (int o = 0; o < 8; ++o)
#pragma unroll
                for (int cc = 0; cc < TM / 2; ++cc) acc2[o][cc] = 0ull;
            // (lanes beyond the last output read the last ones again)
            const int col_a = min(64 * grp + 4 * ql, H - 4), col_b = min(64 * grp + 32 + 4 * ql, H - 4);
            for (int k0 = 0; k0 < in_w; k0 += stage_rows) {
                const int rows = min(stage_rows, in_w - k0);
                ok = __all_sync(0xffffffffu, ok && (next || mbar_wait(smem_u32(full + s), ph, abort_flag)));
                next = mbar_test(smem_u32(full + (s + 1 == lay.stages ? 0 : s + 1)), s + 1 == lay.stages ? ph ^ 1u : ph);
                const T *w0 = reinterpret_cast<const T *>(ring + s * kSimtStageBytes);
                if (ok && busy) {
                    const float *x0 = in_act + k0 * TM;
                    // two rows in registers: the reads of one travel while the other is multiplied
                    struct Row {
                        float4 wa, wb;
                        ulonglong2 xa, xb;
                    } a, bb;
                    const int step = 4 * splits, last = rows - 1;   // reads beyond the stage repeat its last row and are not multiplied
                    auto read = [&](Row &q, int rr) {
                        q.wa = load4(w0 + (size_t)rr * H + col_a), q.wb = load4(w0 + (size_t)rr * H + col_b);
                        q.xa = *reinterpret_cast<const ulonglong2 *>(x0 + rr * TM), q.xb = *reinterpret_cast<const ulonglong2 *>(x0 + rr * TM + 4);
                    };
                    auto multiply = [&](const Row &q) {
                        const uint64_t x[4] = {q.xa.x, q.xa.y, q.xb.x, q.xb.y};
                        const float w[8] = {q.wa.x, q.wa.y, q.wa.z, q.wa.w, q.wb.x, q.wb.y, q.wb.z, q.wb.w};
#pragma unroll
                        for (int o = 0; o < 8; ++o)
#pragma unroll
                            for (int cc = 0; cc < TM / 2; ++cc) acc2[o][cc] = fma_f32x2(pack_f32x2(w[o], w[o]), x[cc], acc2[o][cc]);
                    };
                    int r = kp + 4 * part;
                    read(a, min(r, last));
#pragma unroll 1
                    for (; r + step < rows; r += 2 * step) {
                        read(bb, r + step);
                        multiply(a);
                        read(a, min(r + 2 * step, last));
                        multiply(bb);
                    }
                    if (r < rows) multiply(a);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(empty + s));
                if (++s == lay.stages) s = 0, ph ^= 1u;
            }
            // the four row slices meet: lane (kp, ql) ends with outputs 4 ql + kp and 32 + 4 ql + kp of the warp's 64
            float4 *r = reinterpret_cast<float4 *>(red) + (part * groups + grp) * 128 + 8 * ql;   // unit 2 * output + half, its low bits mixed with ql: no bank conflicts
            const bool hi = kp & 2, odd = kp & 1;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                float v[TM];
#pragma unroll
                for (int cc = 0; cc < TM / 2; ++cc) {
                    float a[4][2], h[2][2];
#pragma unroll
                    for (int o = 0; o < 4; ++o) unpack_f32x2(acc2[4 * g + o][cc], a[o][0], a[o][1]);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
#pragma unroll
                        for (int o = 0; o < 2; ++o) h[o][e] = (hi ? a[2 + o][e] : a[o][e]) + __shfl_xor_sync(0xffffffffu, hi ? a[o][e] : a[2 + o][e], 16);
                        v[2 * cc + e] = (odd ? h[1][e] : h[0][e]) + __shfl_xor_sync(0xffffffffu, odd ? h[0][e] : h[1][e], 8);
                    }
                }
                if (busy) {
                    r[64 * g + ((2 * kp) ^ ql)] = make_float4(v[0], v[1], v[2], v[3]);
                    r[64 * g + ((2 * kp + 1) ^ ql)] = make_float4(v[4], v[5], v[6], v[7]);
                }
            }
            // ... and those of the warps: [part][group][64 outputs][TM], every thread sums outputs of its own
            const int first = tid >> 1;
            const float b_first = first < H ? bias[first] : 0.f;
            named_bar_sync(1, kSimtThreads);
            for (int i = tid; i < 2 * H; i += kSimtThreads) {
                const int o = i >> 1, h = i & 1;
                const float b0 = o == first ? b_first : bias[o];
                float4 v = make_float4(b0, b0, b0, b0);
#pragma unroll 4
                for (int q = 0; q < splits; ++q) {
                    const float4 t = reinterpret_cast<const float4 *>(red)[q * groups * 128 + (i ^ (i >> 3 & 7))];
                    v.x += t.x, v.y += t.y, v.z += t.z, v.w += t.w;
                }
                *reinterpret_cast<float4 *>(out_act + (size_t)o * TM + 4 * h) =
                    make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
            }
        }
        in_act = out_act;
        out_act = (out_act == ha) ? hb : ha;
        in_w = H;
    }
    const T *wo = reinterpret_cast<const T *>(md.w_out);
    float w_first[4];   // requested before the barrier
#pragma unroll
    for (int u = 0; u < 4; ++u) w_first[u] = lane + 32 * u < in_w ? to_f(wo[lane + 32 * u]) : 0.f;
    const bool bad = named_bar_or(1, kSimtThreads, !ok);
    // ---- output layer: warp c reduces candidate c in a fixed order
    if (c < cnt) {
        float acc = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (lane + 32 * u < in_w) acc = fmaf(w_first[u], in_act[(lane + 32 * u) * TM + c], acc);
        for (int j = lane + 128; j < in_w; j += 32) acc = fmaf(to_f(wo[j]), in_act[j * TM + c], acc);
        acc = warp_sum(acc);
        if (lane == 0) {
            float logit = acc + b_out;
            if (md.emit_sigmoid) logit = 1.0f / (1.0f + expf(-logit));
            sl.logits[rq.off + start + c] = id >= 0 && !bad ? logit : __int_as_float(0x7fc00000);
        }
    }
    if (bad) {   // a wait that ran out: copies in flight land before shared memory goes away
        if (tid == 0) atomicOr(sl.status, AIF_STATUS_TIMEOUT);
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) __nanosleep(1000);
    }
}

cudaError_t launch_score_simt(const aif_ctx *ctx, const ScoreLaunch &sl, cudaStream_t st)
{
    if (sl.n_tiles <= 0) return cudaSuccess;
    const aif_config &c = ctx->cfg;
    SimtLayout lay{};
    for (int k = 0; k < c.n_hidden; ++k) lay.max_h = c.hidden[k] > lay.max_h ? c.hidden[k] : lay.max_h;
    const int k1 = ctx->input_width - c.d, act = 2 * lay.max_h * kSimtTile;
    const int chunk = kSimtKeys * (int)(c.d * ctx->el + 16) / 4;
    auto bytes = [&](int stages, int bufs) {
        lay.stages = stages, lay.key_bufs = bufs, lay.region = act > bufs * chunk ? act : bufs * chunk;
        lay.red = stages ? kSimtRed : 0, lay.ps = bufs ? 2 * kSimtWarps * kSimtKeys : 0;
        return ((size_t)(k1 + c.d) * kSimtTile + lay.region + lay.red + lay.ps + (size_t)kSimtTile * (8 + 16)) * 4 +
               (stages ? 64 + (size_t)kSimtMaxStages * 16 + (size_t)stages * kSimtStageBytes : 0);
    };
    // The ring pays where there are weights enough to stream: below 65536 of them a thread per output is as fast in a small launch (96 ->
    // 64 -> 32 units, 1000 candidates: 9.5 against 9.1 us), and three blocks per SM are faster in a large one, to which the ring leaves
    // one (64000 candidates: 184 against 393 us; 256 -> 192 -> 64 units: 600 against 805).  At 98304 (256 -> 256 -> 128 units) 1000
    // candidates take 16.8 us with it.  Layers of more than 256 units: 1000 candidates, 1024 -> 1024 -> 512 -> 256 units, 205 us without, 346
    // with.  Not by the number of candidates: the two sum in different orders, and a logit does not depend on how many share its call.
    int64_t n_weights = 0;
    for (int k = 0; k < c.n_hidden; ++k) n_weights += (int64_t)(k ? c.hidden[k - 1] : k1) * c.hidden[k];
    size_t smem = 0;
    int mode = SIMT_DIRECT;
    if (lay.max_h <= kSimtRingH && n_weights >= kSimtRingWeights) {
        // wide inputs leave less room: for key buffers and stages first, then for none of the ring
        static const int tries[][2] = {{4, 2}, {4, 1}, {3, 1}, {2, 1}};
        for (const auto &t : tries)
            if ((smem = bytes(t[0], t[1])) <= 227 * 1024) {
                mode = SIMT_RING;
                break;
            }
    }
    if (mode != SIMT_RING) {
        // key chunks as there is room for them, three blocks per SM where that is possible
        if ((smem = bytes(0, 2)) > 75 * 1024 && (smem = bytes(0, 1)) > 227 * 1024) smem = bytes(0, 0);
        // up to two blocks per SM the loads of one are what counts (256 -> 512 -> 256 units, 1000 candidates: 71 against 174 us), beyond that
        // the blocks beside each other (32000 candidates: 1886 against 1531), unless their inputs leave room for one only
        // (1024 units and more use three all the same: the layers' reads wait less than they do side by side)
        if (sl.n_tiles > 2 * 148 && (smem <= 113 * 1024 || lay.max_h > kSimtRingH)) mode = SIMT_MANY;
    }
    const ModelDev md = make_model(ctx);
    timing_begin(ctx, st);
    auto go = [&](auto kernel) {
        const cudaError_t e = smem <= 48 * 1024 ? cudaSuccess : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return e != cudaSuccess ? e : launch_pdl(kernel, dim3(sl.n_tiles), dim3(kSimtThreads + (mode == SIMT_RING ? 32 : 0)), smem, st, md, sl, lay);
    };
    const bool f32 = c.dtype == AIF_F32;
    const cudaError_t e = mode == SIMT_RING     ? (f32 ? go(k_score_simt<float, SIMT_RING>) : go(k_score_simt<__nv_bfloat16, SIMT_RING>))
                          : mode == SIMT_DIRECT ? (f32 ? go(k_score_simt<float, SIMT_DIRECT>) : go(k_score_simt<__nv_bfloat16, SIMT_DIRECT>))
                                                : (f32 ? go(k_score_simt<float, SIMT_MANY>) : go(k_score_simt<__nv_bfloat16, SIMT_MANY>));
    count_launch();
    timing_mark(ctx, "score_simt", st);
    return e;
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
