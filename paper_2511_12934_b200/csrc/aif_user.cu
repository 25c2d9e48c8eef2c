// User side of a request (Section 3.1 eqs. 1-3, Section 3.3 "User-Side Pre-Processing", Algorithm 1 steps 1-2), run on a
// side stream in parallel with retrieval.  A user is one request's worth of work, a few tens of MFLOP: what counts is the
// number of launches in a row and the length of the dependent chain inside each, not throughput.  Five launches, each
// started while its predecessor runs out (programmatic dependent launch):
//   1 k_slot_begin   the caller's tensors into the slot (cross pre-cache, V, signatures and their +-1 form, zero padding), the
//                    slot's length; Algorithm 1's V from bea_U, one block per bridge beside the copies
//   2 k_user_gemm    eq. 1: S = seq W_seq^T with the largest row norm, and the projected profile
//   3 k_att_tc       eq. 2's attention rows softmax(S S^T / sqrt(d)) S (aif_tc_att.cu)
//   4 k_user_pool    eq. 2's hidden FFN layer, summed over the sequence; beside it eq. 3 over slices of the keys
//   5 k_user_finish  merges the slices, second FFN layer, the combined vector u, p_u = W1[:, user columns] u + b1
// fp32 storage and widths the warp-level products do not cover take CUDA-core kernels for 2-4.
#include "aif_device.cuh"
#include "aif_internal.h"
#include "aif_tc_ptx.cuh"

namespace aif {
namespace {

// ------------------------------------------------------------------------------------------------
// 1: the slot
// ------------------------------------------------------------------------------------------------
// One contiguous piece of a slot in units of 16 bytes: copied from src, zeroed (src == nullptr), or expanded (two signature
// bytes of src -> sixteen +-1 bytes).
struct SlotPiece {
    const void *src;
    void *dst;
    int64_t units;
    int32_t expand;
};
constexpr int kMaxPieces = 8;
struct SlotPieces {
    SlotPiece p[kMaxPieces];
    int32_t n;
    int64_t units;   // of all pieces
};

struct BeaUser {
    const void *Bm, *U, *Wf;
    void *V;
    int32_t n, m, d;   // n: bridges, one block each (0: none)
};

// Algorithm 1 steps 1-2 for bridge k, by one block: w = softmax(B_k U^T / sqrt(d)), A = sum_j w_j U_j, V_k = W_f A.
template <typename T>
__device__ void bea_bridge(const BeaUser &b, int k, float *sm)
{
    const T *Bm = (const T *)b.Bm + (size_t)k * b.d, *U = (const T *)b.U, *Wf = (const T *)b.Wf;
    const int d = b.d, m = b.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *W = sm, *A = W + m, *red = A + d;   // [m], [d], [256]
    const float scale = rsqrtf((float)d);
    for (int j0 = warp * 4; j0 < m; j0 += 32) {   // four features per warp and round: their loads are in flight together
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int c = lane; c < d; c += 32) {
            const float q = to_f(Bm[c]);
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = fmaf(q, to_f(U[(size_t)min(j0 + u, m - 1) * d + c]), acc[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            acc[u] = warp_sum(acc[u]);
            if (lane == 0 && j0 + u < m) W[j0 + u] = acc[u] * scale;
        }
    }
    __syncthreads();
    float mx = -INFINITY, den = 0.f;   // every warp takes the same maximum and sum over the m scores
    for (int j = lane; j < m; j += 32) mx = fmaxf(mx, W[j]);
    mx = warp_max(mx);
    for (int j = lane; j < m; j += 32) den += expf(W[j] - mx);
    den = warp_sum(den);
    {
        const int parts = 256 / d, c = tid % d, part = tid / d;   // d <= 256
        float acc = 0.f;
        if (part < parts)
#pragma unroll 8
            for (int j = part; j < m; j += parts) acc = fmaf(expf(W[j] - mx) / den, to_f(U[(size_t)j * d + c]), acc);
        red[tid] = acc;
        __syncthreads();
        if (tid < d) {
            float a = 0.f;
            for (int q = 0; q < parts; ++q) a += red[q * d + tid];
            A[tid] = a;
        }
    }
    __syncthreads();
    for (int r0 = warp * 4; r0 < d; r0 += 32) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int c = lane; c < d; c += 32) {
            const float a = A[c];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u] = fmaf(to_f(Wf[(size_t)(r0 + u) * d + c]), a, acc[u]);   // d is a multiple of 32
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            acc[u] = warp_sum(acc[u]);
            if (lane == 0) from_f(((T *)b.V)[(size_t)k * d + r0 + u], acc[u]);
        }
    }
}

// Copies run at memory speed over all SMs; the blocks of the bridges come first, so that their chain of dependent steps runs
// beside the copies.  One block for all bridges took 90 us at 8 bridges and 64 features.
template <typename T>
__global__ void __launch_bounds__(256) k_slot_begin(SlotPieces sp, BeaUser bea, SlotDev *slots, int index, int L)
{
    extern __shared__ float sm_bea[];
    grid_dep_launch();
    grid_dep_wait();
    if ((int)blockIdx.x < bea.n) {
        bea_bridge<T>(bea, blockIdx.x, sm_bea);
        return;
    }
    const int64_t block = (int64_t)blockIdx.x - bea.n, n_blocks = (int64_t)gridDim.x - bea.n;
    if (block == 0 && threadIdx.x == 0) {
        slots[index].L = L;
        *const_cast<float *>(slots[index].k_norm) = 0.f;   // raised by whoever writes the rows of S
    }
    const int64_t stride = n_blocks * 256;
    for (int64_t i = block * 256 + threadIdx.x; i < sp.units; i += 4 * stride) {
        uint4 v[4];
        uint4 *dst[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int64_t k = i + u * stride;
            dst[u] = nullptr;
            if (k >= sp.units) continue;
            int q = 0;
            while (k >= sp.p[q].units) k -= sp.p[q++].units;
            dst[u] = (uint4 *)sp.p[q].dst + k;
            if (!sp.p[q].src) v[u] = make_uint4(0, 0, 0, 0);
            else if (!sp.p[q].expand) v[u] = __ldg((const uint4 *)sp.p[q].src + k);
            else {
                const uint32_t two = __ldg((const uint16_t *)sp.p[q].src + k);
                v[u] = expand_sig16(two & 0xFFu, two >> 8);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (dst[u]) *dst[u] = v[u];
    }
}

// ------------------------------------------------------------------------------------------------
// 2, 4: products over the sequence rows on the warp-level matrix instructions
// ------------------------------------------------------------------------------------------------
// [rows x K] . [K x N] with K = 32 VJ and N = 64 NT: a block of eight warps takes 16 rows at a time, every warp 8 NT output
// columns, its slice of the weights in registers for the whole launch.  The order of K inside a product is free, so both
// operands are read 16 contiguous bytes per thread straight from global memory, all of them in flight at once: no shared
// memory, no pipeline to fill, one memory latency per 16 rows.  A tcgen05 tile needs 128 rows, tensor memory and a weight
// ring set up before its first product; at the 50 to 10^4 rows of one user that costs more than the product.
// (K, N) of one thread's fragments: lane 4 g + t holds rows g, g + 8 and columns 2 t, 2 t + 1 of every eight.
template <int VJ, int NT>
struct WeightSlice {
    uint4 b[NT][VJ];
    // W [N x K] row-major; the eight columns of slice j of this warp start at n0 + 8 j
    __device__ __forceinline__ void load(const __nv_bfloat16 *W, int n0, int g, int t)
    {
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int v = 0; v < VJ; ++v) b[j][v] = __ldg(reinterpret_cast<const uint4 *>(W + (size_t)(n0 + 8 * j + g) * (32 * VJ) + 8 * (t + 4 * v)));
    }
    __device__ __forceinline__ void product(float (&c)[NT][4], const __nv_bfloat16 *row_lo, const __nv_bfloat16 *row_hi, int t) const
    {
        uint4 lo[VJ], hi[VJ];
#pragma unroll
        for (int v = 0; v < VJ; ++v) {
            lo[v] = *reinterpret_cast<const uint4 *>(row_lo + 8 * (t + 4 * v));
            hi[v] = *reinterpret_cast<const uint4 *>(row_hi + 8 * (t + 4 * v));
        }
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            c[j][0] = c[j][1] = c[j][2] = c[j][3] = 0.f;
#pragma unroll
            for (int v = 0; v < VJ; ++v) {
                mma_bf16(c[j], lo[v].x, hi[v].x, lo[v].y, hi[v].y, b[j][v].x, b[j][v].y);
                mma_bf16(c[j], lo[v].z, hi[v].z, lo[v].w, hi[v].w, b[j][v].z, b[j][v].w);
            }
        }
    }
};

// eq. 1.  Blocks 0 .. gridDim.x - 2: rows of S; the last block: the profile as a one-row product with W_profile.
template <int VJ, int NT>
__global__ void __launch_bounds__(256) k_user_gemm(const __nv_bfloat16 *__restrict__ seq, const __nv_bfloat16 *__restrict__ profile,
                                                   const __nv_bfloat16 *__restrict__ Wseq, const __nv_bfloat16 *__restrict__ Wprof, int L,
                                                   __nv_bfloat16 *__restrict__ S, float *__restrict__ prof_hat, float *__restrict__ k_norm)
{
    constexpr int K = 32 * VJ, N = 64 * NT;
    __shared__ float ss_s[8][16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3, n0 = warp * 8 * NT;
    const bool is_prof = blockIdx.x == gridDim.x - 1;
    grid_dep_launch();
    WeightSlice<VJ, NT> w;
    w.load(is_prof ? Wprof : Wseq, n0, g, t);   // weights are older than any launch this one may overlap
    grid_dep_wait();
    float c[NT][4];
    if (is_prof) {
        w.product(c, profile, profile, t);
        if (g == 0)
#pragma unroll
            for (int j = 0; j < NT; ++j) prof_hat[n0 + 8 * j + 2 * t] = c[j][0], prof_hat[n0 + 8 * j + 2 * t + 1] = c[j][1];
        return;
    }
    int best = 0;
    for (int i0 = blockIdx.x * 16; i0 < L; i0 += (gridDim.x - 1) * 16) {
        const int r[2] = {i0 + g, i0 + g + 8};
        w.product(c, seq + (size_t)min(r[0], L - 1) * K, seq + (size_t)min(r[1], L - 1) * K, t);
        float ss[2] = {0.f, 0.f};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const __nv_bfloat162 o = __floats2bfloat162_rn(c[j][2 * h], c[j][2 * h + 1]);
                const float2 f = __bfloat1622float2(o);
                ss[h] = fmaf(f.x, f.x, fmaf(f.y, f.y, ss[h]));
                if (r[h] < L) *reinterpret_cast<__nv_bfloat162 *>(S + (size_t)r[h] * N + n0 + 8 * j + 2 * t) = o;
            }
            ss[h] += __shfl_xor_sync(0xffffffffu, ss[h], 1);
            ss[h] += __shfl_xor_sync(0xffffffffu, ss[h], 2);
            if (t == 0) ss_s[warp][g + 8 * h] = ss[h];
        }
        __syncthreads();
        if (warp == 0 && lane < 16 && i0 + lane < L) {
            float a = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) a += ss_s[q][lane];
            best = max(best, __float_as_int(sqrtf(a)) & 0x7fffffff);   // norms order like their bit patterns, NaN above all
        }
        __syncthreads();
    }
    if (warp == 0) {
        best = __reduce_max_sync(0xffffffffu, best);
        if (lane == 0 && best > 0) atomicMax(reinterpret_cast<int *>(k_norm), best);
    }
}

__device__ __forceinline__ void load8(const __nv_bfloat16 *p, float (&f)[8])
{
    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 a = __bfloat1622float2(h[i]);
        f[2 * i] = a.x, f[2 * i + 1] = a.y;
    }
}
__device__ __forceinline__ void load8(const float *p, float (&f)[8])
{
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p)), b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    f[0] = a.x, f[1] = a.y, f[2] = a.z, f[3] = a.w, f[4] = b.x, f[5] = b.y, f[6] = b.z, f[7] = b.w;
}

// eq. 3 over keys [start, start + len) by one warp: LPR lanes own eight columns each of a key row, 32 / LPR rows per load and
// eight loads per step, so a step's keys are fetched once, together, and serve both the scores and the weighted sum from
// registers.  Leaves the unnormalised row, its maximum and its sum: out[0..d), out[d], out[d + 1].
template <typename T, int LPR>
__device__ __forceinline__ void profile_slice(const T *__restrict__ S, int start, int len, const float *__restrict__ prof_hat, int d,
                                              float *__restrict__ out)
{
    constexpr int RPI = 32 / LPR;
    const int lane = threadIdx.x & 31, sub = lane / LPR, c = (lane % LPR) * 8;
    const bool own = c < d;   // d need not fill the lanes
    const float scale = rsqrtf((float)d);
    float q[8], acc[8], m = -INFINITY, l = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = 0.f, acc[i] = 0.f;
    if (own) load8(prof_hat + c, q);
    for (int j0 = 0; j0 < len; j0 += 8 * RPI) {
        float v[8][8], s[8], mx = m;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int r = min(j0 + u * RPI + sub, len - 1);
#pragma unroll
            for (int i = 0; i < 8; ++i) v[u][i] = 0.f;
            if (own) load8(S + (size_t)(start + r) * d + c, v[u]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            s[u] = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) s[u] = fmaf(q[i], v[u][i], s[u]);
#pragma unroll
            for (int o = LPR / 2; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
            s[u] = j0 + u * RPI + sub < len ? s[u] * scale : -INFINITY;
            mx = fmaxf(mx, s[u]);
        }
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float off = mx == -INFINITY ? 0.f : mx;   // nothing but scores of minus infinity so far: no weight
        const float f = expf(m - off);
        m = mx, l *= f;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] *= f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float p = expf(s[u] - off);
            l += p;
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = fmaf(p, v[u][i], acc[i]);
        }
    }
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) {
        l += __shfl_xor_sync(0xffffffffu, l, o);
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
    }
    if (sub == 0 && own) {
        reinterpret_cast<float4 *>(out + c)[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        reinterpret_cast<float4 *>(out + c)[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    if (lane == 0) out[d] = m, out[d + 1] = l;
}

template <typename T>
__device__ __forceinline__ void profile_slices(const T *S, int L, int d, const float *prof_hat, int slice, int n_slices, int block, float *ppart)
{
    const int g = block * 8 + (threadIdx.x >> 5), start = g * slice;
    if (g >= n_slices) return;
    float *out = ppart + (size_t)g * (d + 4);
    const int len = min(slice, L - start);
    if (d <= 64) profile_slice<T, 8>(S, start, len, prof_hat, d, out);
    else if (d <= 128) profile_slice<T, 16>(S, start, len, prof_hat, d, out);
    else profile_slice<T, 32>(S, start, len, prof_hat, d, out);
}

// eq. 2's FFN hidden layer over the attention rows, ReLU(a W_a^T + b_a), summed over the rows of this block's share (the second
// FFN layer is linear, so it commutes with the mean pooling and is applied once, in k_user_finish): partial[block][N].
// Blocks from n_ffn on: eq. 3's key slices, which need nothing of the attention rows.
template <int VJ, int NT>
__global__ void __launch_bounds__(256) k_user_pool(const __nv_bfloat16 *__restrict__ rows, const __nv_bfloat16 *__restrict__ Wa,
                                                   const float *__restrict__ b_a, int L, int n_ffn, float *__restrict__ partial,
                                                   const __nv_bfloat16 *__restrict__ S, const float *__restrict__ prof_hat, int slice,
                                                   int n_slices, float *__restrict__ ppart)
{
    constexpr int K = 32 * VJ, N = 64 * NT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3, n0 = warp * 8 * NT;
    grid_dep_launch();
    if ((int)blockIdx.x >= n_ffn) {
        grid_dep_wait();
        profile_slices<__nv_bfloat16>(S, L, N, prof_hat, slice, n_slices, (int)blockIdx.x - n_ffn, ppart);
        return;
    }
    WeightSlice<VJ, NT> w;
    w.load(Wa, n0, g, t);
    float bias[NT][2], sum[NT][2];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int q = 0; q < 2; ++q) bias[j][q] = b_a[n0 + 8 * j + 2 * t + q], sum[j][q] = 0.f;
    grid_dep_wait();
    for (int i0 = blockIdx.x * 16; i0 < L; i0 += n_ffn * 16) {
        float c[NT][4];
        w.product(c, rows + (size_t)min(i0 + g, L - 1) * K, rows + (size_t)min(i0 + g + 8, L - 1) * K, t);
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (i0 + g + 8 * h < L) {
                    sum[j][0] += fmaxf(c[j][2 * h] + bias[j][0], 0.f);
                    sum[j][1] += fmaxf(c[j][2 * h + 1] + bias[j][1], 0.f);
                }
    }
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float v = sum[j][q];
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (g == 0) partial[(size_t)blockIdx.x * N + n0 + 8 * j + 2 * t + q] = v;
        }
}

// ------------------------------------------------------------------------------------------------
// the same steps on CUDA cores: fp32 storage, and widths the products above do not cover
// ------------------------------------------------------------------------------------------------
// eq. 1.  blockIdx.x < L: one sequence row -> S (storage type).  blockIdx.x == L: the profile -> prof_hat (fp32).
template <typename T>
__global__ void k_user_project(const T *__restrict__ seq, const T *__restrict__ profile, const T *__restrict__ Wseq_t,
                               const T *__restrict__ Wprof_t, int L, int dU, int d, T *__restrict__ S,
                               float *__restrict__ prof_hat)
{
    extern __shared__ float row[];
    const bool is_prof = (int)blockIdx.x == L;
    const T *src = is_prof ? profile : seq + (size_t)blockIdx.x * dU;
    const T *W = is_prof ? Wprof_t : Wseq_t;
    for (int k = threadIdx.x; k < dU; k += blockDim.x) row[k] = to_f(src[k]);
    __syncthreads();
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
        float acc = 0.f;
        for (int k = 0; k < dU; ++k) acc = fmaf(row[k], to_f(W[(size_t)k * d + j]), acc);
        if (is_prof) prof_hat[j] = acc;
        else from_f(S[(size_t)blockIdx.x * d + j], acc);
    }
}

// eq. 2.  Warp g handles rows g, g + n_warps, ...: attention over the whole sequence, FFN hidden layer, running sum; partial[g] holds
// the warp's sum.
template <typename T>
__global__ void __launch_bounds__(256) k_user_self(const T *__restrict__ S, int L, int d, const T *__restrict__ Wa_t,
                                                   const float *__restrict__ b_a, float *__restrict__ partial, int n_warps)
{
    extern __shared__ float sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = blockIdx.x * 8 + warp, dq = d >> 5;
    float *q = sm + (size_t)warp * 2 * d, *ctx = q + d;
    float pooled[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) pooled[c] = 0.f;
    const float scale = rsqrtf((float)d);
    for (int i = g; i < L; i += n_warps) {
        for (int k = lane; k < d; k += 32) q[k] = to_f(S[(size_t)i * d + k]);
        __syncwarp();
        float att[8], din[8];
        warp_interact<T>(q, S, L, d, scale, true, false, false, nullptr, nullptr, 0, 0, nullptr, att, din);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < dq) ctx[lane + 32 * c] = att[c];
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < dq) {
                const int j = lane + 32 * c;
                float acc = b_a[j];
                for (int k = 0; k < d; ++k) acc = fmaf(ctx[k], to_f(Wa_t[(size_t)k * d + j]), acc);
                pooled[c] += fmaxf(acc, 0.f);
            }
        __syncwarp();
    }
    if (g < n_warps) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < dq) partial[(size_t)g * d + lane + 32 * c] = pooled[c];
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_user_prof(const T *__restrict__ S, int L, int d, const float *__restrict__ prof_hat, int slice,
                                                   int n_slices, float *__restrict__ ppart)
{
    profile_slices<T>(S, L, d, prof_hat, slice, n_slices, blockIdx.x, ppart);
}

// ------------------------------------------------------------------------------------------------
// 5: u and p_u
// ------------------------------------------------------------------------------------------------
// raw = 1: u = mean-pooled self-attention through the second FFN layer + profile attention; raw = 0: u is given.  Every block
// forms u for itself (the partial sums it merges are tens of KB in L2) and then kFinishCols entries of p_u, so that the
// chain of dependent steps is not followed by one block's walk over the whole of W1.  Each step on the way to u spreads its loads
// over all threads, a column group of 16 bytes and a slice of the rows per thread, and joins the slices in shared memory in a fixed
// order.  One block over 1184 partial sums, with one column per thread and 2-byte loads, took 66 us at d = 128, H1 = 512.
// p_u itself is one running sum per entry, b1 and then the columns of u in their order, as the first layer defines it: a sum in
// slices moves hidden activations across bf16 rounding edges, and the logits of a three-layer model by 1e-4 of their size.  The
// columns of W1 are brought to shared memory by all threads, under the steps before, so that the chain of d multiply-adds waits for
// nothing else.
constexpr int kFinishCols = 64, kFinishTile = 32768;
template <typename T>
__global__ void __launch_bounds__(256) k_user_finish(int raw, int L, int d, const float *__restrict__ partial, int n_parts,
                                                     const float *__restrict__ ppart, int n_slices, const T *__restrict__ u_in,
                                                     T *__restrict__ u_out, float *__restrict__ u32, const T *__restrict__ Wb_t,
                                                     const float *__restrict__ b_b, const T *__restrict__ W1t, const float *__restrict__ b1,
                                                     int H1, float *__restrict__ p_u, __nv_bfloat16 *__restrict__ pu_hl)
{
    __shared__ __align__(16) float red[2][1024];
    __shared__ float us[256], q_s[256], uprof[256], wgt[kProfParts], wred[8];
    constexpr int kRows = kFinishTile / (kFinishCols * (int)sizeof(T)), kUnits = kFinishCols * (int)sizeof(T) / 16;
    __shared__ __align__(16) T w1_s[kRows * kFinishCols];   // rows k0 .. of this block's columns of W1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, col0 = blockIdx.x * kFinishCols;
    static_assert(kProfParts == 256, "one thread per key slice");
    auto fetch = [&](int k0) {   // 16 bytes at a time: H1 is a multiple of 8; columns beyond it as zeros
        for (int i = tid; i < min(kRows, d - k0) * kUnits; i += 256) {
            const int r = i / kUnits, col = col0 + (i % kUnits) * (16 / (int)sizeof(T));
            cp_async16(smem_u32(w1_s) + i * 16, W1t + (size_t)(k0 + r) * H1 + (col < H1 ? col : 0), col < H1 ? 16u : 0u);
        }
        cp_async_commit();
    };
    grid_dep_launch();
    grid_dep_wait();
    fetch(0);
    if (raw) {
        // weights 2^(m_g - m) of the key slices
        const float m_g = tid < n_slices ? ppart[(size_t)tid * (d + 4) + d] : -INFINITY, l_g = tid < n_slices ? ppart[(size_t)tid * (d + 4) + d + 1] : 0.f;
        float mx = warp_max(m_g);
        if (lane == 0) wred[warp] = mx;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) mx = fmaxf(mx, wred[i]);
        const float w = tid < n_slices ? expf(m_g - mx) : 0.f;
        wgt[tid] = w;
        const float ls = warp_sum(w * l_g);
        __syncthreads();
        if (lane == 0) wred[warp] = ls;
        // both merges: four columns per thread, `parts` threads per column group over interleaved slices
        const int groups = d / 4, parts = 256 / groups, cg = tid % groups, part = tid / groups;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (part < parts) {
#pragma unroll 8
            for (int i = part; i < n_slices; i += parts) {
                const float4 v = *reinterpret_cast<const float4 *>(ppart + (size_t)i * (d + 4) + 4 * cg);
                const float wi = wgt[i];
                a.x = fmaf(wi, v.x, a.x), a.y = fmaf(wi, v.y, a.y), a.z = fmaf(wi, v.z, a.z), a.w = fmaf(wi, v.w, a.w);
            }
#pragma unroll 8
            for (int i = part; i < n_parts; i += parts) {
                const float4 v = *reinterpret_cast<const float4 *>(partial + (size_t)i * d + 4 * cg);
                b.x += v.x, b.y += v.y, b.z += v.z, b.w += v.w;
            }
            reinterpret_cast<float4 *>(red[0])[part * groups + cg] = a;
            reinterpret_cast<float4 *>(red[1])[part * groups + cg] = b;
        }
        __syncthreads();
        if (tid < d) {
            float den = 0.f, pa = 0.f, pb = 0.f;
            for (int i = 0; i < 8; ++i) den += wred[i];
            for (int i = 0; i < parts; ++i) pa += red[0][i * d + tid], pb += red[1][i * d + tid];
            uprof[tid] = pa / den;
            q_s[tid] = pb / (float)L;
        }
        __syncthreads();
        // the second FFN layer of the pooled row
        const int g8 = d / 8, p8 = 256 / g8, c8 = (tid % g8) * 8, r8 = tid / g8;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (r8 < p8) {
#pragma unroll 8
            for (int k = r8; k < d; k += p8) {
                float f[8];
                load8(Wb_t + (size_t)k * d + c8, f);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = fmaf(q_s[k], f[i], acc[i]);
            }
            float *o = red[0] + r8 * d + c8;   // p8 x d <= 2048 floats: both halves of red
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] = acc[i];
        }
        __syncthreads();
        if (tid < d) {
            float u = b_b[tid];
            for (int i = 0; i < p8; ++i) u += red[0][i * d + tid];
            u += uprof[tid];
            us[tid] = u;
            if (blockIdx.x == 0) {
                u32[tid] = u;
                from_f(u_out[tid], u);
            }
        }
    } else if (tid < d) {
        us[tid] = to_f(u_in[tid]);
        if (blockIdx.x == 0) u32[tid] = us[tid];
    }
    const int j = col0 + tid;
    const bool own = tid < kFinishCols && j < H1;
    float acc = own ? b1[j] : 0.f;
    for (int k0 = 0; k0 < d; k0 += kRows) {
        if (k0) {
            __syncthreads();
            fetch(k0);
        }
        cp_async_wait<0>();
        __syncthreads();   // (and us)
        if (tid < kFinishCols)
#pragma unroll 16
            for (int k = 0; k < min(kRows, d - k0); ++k) acc = fmaf(us[k0 + k], to_f(w1_s[k * kFinishCols + tid]), acc);
    }
    if (own) {
        p_u[j] = acc;
        // the same partial as two bf16 values (high part, remainder): the form in which the tensor cores add it
        const __nv_bfloat16 hi = __float2bfloat16_rn(acc);
        pu_hl[j] = hi;
        pu_hl[H1 + j] = __float2bfloat16_rn(acc - __bfloat162float(hi));
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
using bf16 = __nv_bfloat16;

// Widths of the warp-level products: K in {64, 128, 256} (16-byte pieces of a quad), N in {64, 128, 256} (eight warps of whole
// eight-column slices, the weight slice in registers).
bool mma_width(int v) { return v == 64 || v == 128 || v == 256; }

cudaError_t launch_gemm(const aif_ctx *ctx, const HostSlot &hs, const aif_user_inputs *in, int L, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    const int tiles = (L + 15) / 16, grid = (tiles < 592 ? tiles : 592) + 1;
    auto go = [&](auto kernel) {
        return launch_pdl(kernel, dim3(grid), dim3(256), 0, st, (const bf16 *)in->seq, (const bf16 *)in->profile, (const bf16 *)ctx->Wseq_k,
                          (const bf16 *)ctx->Wprof_k, L, (bf16 *)hs.dev.S, hs.prof_hat, const_cast<float *>(hs.dev.k_norm));
    };
    auto by_n = [&](auto k1, auto k2, auto k4) { return c.d == 64 ? go(k1) : c.d == 128 ? go(k2) : go(k4); };
    count_launch();
    if (c.dU == 64) return by_n(k_user_gemm<2, 1>, k_user_gemm<2, 2>, k_user_gemm<2, 4>);
    if (c.dU == 128) return by_n(k_user_gemm<4, 1>, k_user_gemm<4, 2>, k_user_gemm<4, 4>);
    return by_n(k_user_gemm<8, 1>, k_user_gemm<8, 2>, k_user_gemm<8, 4>);
}

cudaError_t launch_pool(const aif_ctx *ctx, const HostSlot &hs, const void *att_rows, int L, int n_ffn, int slice, int n_slices, cudaStream_t st)
{
    const int d = ctx->cfg.d, grid = n_ffn + (n_slices + 7) / 8;
    auto go = [&](auto kernel) {
        return launch_pdl(kernel, dim3(grid), dim3(256), 0, st, (const bf16 *)att_rows, (const bf16 *)ctx->Wa_k, (const float *)ctx->b_a, L, n_ffn,
                          hs.partial, (const bf16 *)hs.dev.S, (const float *)hs.prof_hat, slice, n_slices, hs.ppart);
    };
    count_launch();
    return d == 128 ? go(k_user_pool<4, 2>) : go(k_user_pool<8, 4>);
}

template <typename T>
cudaError_t user_network_typed(const aif_ctx *ctx, HostSlot &hs, int slot_index, const aif_user_inputs *in, int L, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    const int d = c.d, H1 = c.hidden[0];
    const bool raw = in->mode == AIF_USER_RAW;
    const bool lsh = c.blocks & (AIF_BLK_LSH_DIN | AIF_BLK_SIMTIER);
    cudaError_t e = cudaSuccess;
    T *S = (T *)hs.dev.S;

    // ---- 1: what the slot takes over as it is
    SlotPieces sp{};
    auto add = [&](const void *src, void *dst, int64_t units, int expand) {
        if (units <= 0) return;
        sp.p[sp.n++] = SlotPiece{src, dst, units, expand};
        sp.units += units;
    };
    auto copy = [&](const void *dst, const void *src, size_t bytes) {
        if (bytes % 16 == 0 && (uintptr_t)src % 16 == 0) add(src, const_cast<void *>(dst), (int64_t)(bytes / 16), 0);
        else if (e == cudaSuccess) e = cudaMemcpyAsync(const_cast<void *>(dst), src, bytes, cudaMemcpyDeviceToDevice, st);
    };
    if (c.blocks & AIF_BLK_CROSS) copy(hs.dev.T, in->cross_raw, (size_t)c.F * c.B * c.dc * ctx->el);
    if (!raw) {
        copy(S, in->seq, (size_t)L * d * sizeof(T));
        copy(hs.dev.u, in->profile, (size_t)d * sizeof(T));
    }
    // block-wise readers see zero rows from the end of the sequence to the end of its last 128-key block
    const int L_pad = (L + 127) / 128 * 128 < c.L_max ? (L + 127) / 128 * 128 : c.L_max;
    add(nullptr, S + (size_t)L * d, (int64_t)(L_pad - L) * d * (int64_t)sizeof(T) / 16, 0);
    if (lsh) {
        copy(hs.dev.sigS, in->seq_sig, (size_t)L * (c.lsh_bits / 8));
        if (ctx->tc_lsh_plan) {   // the form the tensor-core LSH kernel multiplies: one +-1 byte per signature bit
            uint8_t *out = const_cast<uint8_t *>(hs.dev.sigE);
            // (an odd address cannot be read two bytes at a time: from the slot's own copy then, which is already queued)
            add((uintptr_t)in->seq_sig % 2 ? hs.dev.sigS : in->seq_sig, out, (int64_t)L * (c.lsh_bits / 16), 1);
            add(nullptr, out + (size_t)L * c.lsh_bits, (int64_t)(L_pad - L) * c.lsh_bits / 16, 0);
        }
    }
    BeaUser bea{};
    if ((c.blocks & AIF_BLK_BEA) && in->bea_V) copy(hs.dev.V, in->bea_V, (size_t)c.n_bridge * d * ctx->el);
    else if (c.blocks & AIF_BLK_BEA) bea = BeaUser{ctx->bridges, in->bea_U, ctx->W_f, const_cast<void *>(hs.dev.V), c.n_bridge, in->bea_m, d};
    if (e != cudaSuccess) return e;
    const int64_t want = (sp.units + 1023) / 1024;
    const int grid = (int)(want < 1 ? 1 : want < 148 * 8 ? want : 148 * 8) + bea.n;
    e = launch_pdl(k_slot_begin<T>, dim3(grid), dim3(256), bea.n ? (size_t)(bea.m + d + 256) * 4 : 0, st, sp, bea, ctx->slots_dev, slot_index, L);
    count_launch();
    if (e != cudaSuccess) return e;

    // ---- 2 to 4
    int n_parts = 0, n_slices = 0;
    if (raw) {
        const bool bf = c.dtype == AIF_BF16;
        if (bf && mma_width(c.dU) && mma_width(d) && (uintptr_t)in->seq % 16 == 0 && (uintptr_t)in->profile % 16 == 0) {
            if ((e = launch_gemm(ctx, hs, in, L, st)) != cudaSuccess) return e;
        } else {
            k_user_project<T><<<L + 1, 128, c.dU * sizeof(float), st>>>((const T *)in->seq, (const T *)in->profile, (const T *)ctx->Wseq_t,
                                                                        (const T *)ctx->Wprofile_t, L, c.dU, d, S, hs.prof_hat);
            count_launch();
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if ((e = launch_row_norm_max(ctx, S, L, const_cast<float *>(hs.dev.k_norm), st)) != cudaSuccess) return e;
        }
        const void *att_rows = nullptr;   // eq. 2: the attention rows on the tensor cores where the shape allows (d = 128, 256), else in k_user_self
        if (bf && ctx->tc_att_plan && (e = launch_self_att_tc(ctx, slot_index, L, st, &att_rows)) != cudaSuccess) return e;
        // key slices of eq. 3: whole steps of a warp (256 / d rows per load, eight loads), at most kProfParts of them
        const int step = 8 * (d <= 64 ? 4 : d <= 128 ? 2 : 1);
        const int slice = ((L + kProfParts - 1) / kProfParts + step - 1) / step * step;
        n_slices = (L + slice - 1) / slice;
        if (att_rows) {
            n_parts = (L + 15) / 16 < 148 ? (L + 15) / 16 : 148;
            if ((e = launch_pool(ctx, hs, att_rows, L, n_parts, slice, n_slices, st)) != cudaSuccess) return e;
        } else {
            k_user_prof<T><<<(n_slices + 7) / 8, 256, 0, st>>>(S, L, d, hs.prof_hat, slice, n_slices, hs.ppart);
            n_parts = (L + 7) / 8 * 8 < kUserPartials ? (L + 7) / 8 * 8 : kUserPartials;
            k_user_self<T><<<n_parts / 8, 256, 8 * 2 * d * sizeof(float), st>>>(S, L, d, (const T *)ctx->Wa_t, ctx->b_a, hs.partial, n_parts);
            count_launch(2);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    } else if ((e = launch_row_norm_max(ctx, S, L, const_cast<float *>(hs.dev.k_norm), st)) != cudaSuccess)
        return e;

    // ---- 5
    e = launch_pdl(k_user_finish<T>, dim3((H1 + kFinishCols - 1) / kFinishCols), dim3(256), 0, st, raw ? 1 : 0, L, d, (const float *)hs.partial,
                   n_parts, (const float *)hs.ppart, n_slices, (const T *)in->profile, (T *)hs.dev.u, (float *)hs.dev.u32, (const T *)ctx->Wb_t,
                   (const float *)ctx->b_b, (const T *)ctx->Wt[0], (const float *)ctx->b[0], H1, (float *)hs.dev.p_u, (bf16 *)hs.dev.pu_hl);
    count_launch();
    return e;
}

}  // namespace

cudaError_t launch_user_network(const aif_ctx *ctx, HostSlot &hs, int slot_index, const aif_user_inputs *in, int L, cudaStream_t st)
{
    if (ctx->cfg.dtype == AIF_F32) return user_network_typed<float>(ctx, hs, slot_index, in, L, st);
    return user_network_typed<bf16>(ctx, hs, slot_index, in, L, st);
}

}  // namespace aif
