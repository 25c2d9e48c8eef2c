// What the two kernels that score a whole request in one launch have in common (aif_tc_fused.cu: a tile per CTA, aif_tc_split.cu: a tile per
// cluster): the attention of a tile and the addresses of its cross features.  A candidate's logit is the same bits by either, so
// what is computed per candidate stands here once.
//
// The softmax and epilogue warps are two groups of four (256 threads, named barrier 1); a thread owns a candidate's row (tensor-memory lane), group
// g the keys [128 g, 128 g + 128).  Tensor memory: scores [0, 256), O [256, 384), probabilities [384, 512) as packed bf16.
#pragma once

#include "aif_device.cuh"
#include "aif_internal.h"
#include "aif_tc_ptx.cuh"

namespace aif {
namespace {

struct RequestRow {
    uint32_t lane_base;   // tensor memory, this warp's lanes
    int g, row;
    int valid_cols;       // keys of the sequence among the group's
    bool act;             // the group has keys and the warp has rows
    float k2;             // log2(e) / sqrt(d)
};

// P = 2^(s k2 - mt) as packed bf16; returns the row sum over the group's keys.
__device__ __forceinline__ float request_probabilities(const RequestRow &r, float mt)
{
    float lsum = 0.f;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        uint32_t sc[64];
        tmem_ld32(r.lane_base + (uint32_t)(r.g * 128 + 64 * h), *reinterpret_cast<uint32_t(*)[32]>(&sc[0]));
        tmem_ld32(r.lane_base + (uint32_t)(r.g * 128 + 64 * h + 32), *reinterpret_cast<uint32_t(*)[32]>(&sc[32]));
        tmem_ld_wait();
        uint32_t packed[32];
        float ls4[4] = {0.f, 0.f, 0.f, 0.f};
        const int left = r.valid_cols - 64 * h;   // valid columns among these 64
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float p0 = fast_exp2(fmaf(__uint_as_float(sc[2 * i]), r.k2, -mt));
            float p1 = fast_exp2(fmaf(__uint_as_float(sc[2 * i + 1]), r.k2, -mt));
            if (2 * i >= left) p0 = 0.f;
            if (2 * i + 1 >= left) p1 = 0.f;
            ls4[i & 3] += p0 + p1;
            const __nv_bfloat162 hh = __floats2bfloat162_rn(p0, p1);
            packed[i] = *reinterpret_cast<const uint32_t *>(&hh);
        }
        tmem_st32(r.lane_base + 384u + (uint32_t)(r.g * 64 + 32 * h), packed);
        lsum += (ls4[0] + ls4[1]) + (ls4[2] + ls4[3]);
    }
    tmem_st_wait();
    return lsum;
}

// Scores -> probabilities; returns the row's sum over all keys.  Softmax is invariant to the offset subtracted in the exponent, and bf16 keeps its
// relative precision over the whole fp32 exponent range.  The first attempt therefore subtracts nothing, p = 2^(s k2), and saves the pass over the
// scores that finds the row maxima; a row sum outside [2^-80, 2^80] (scores far from zero: overflow, or every term flushed to zero) makes the
// whole CTA repeat the step with the exact row maxima.  The probabilities go to columns of their own, so the scores are still there for the
// repeat.  ROWS rows at most: xs[2][ROWS] takes what the groups hand each other; counts: the row is a candidate's place.
template <int ROWS, typename WaitScores>
__device__ __forceinline__ float request_softmax(const RequestRow &r, float *xs, const bool &ok, bool counts, WaitScores wait_scores)
{
    const int g = r.g, row = r.row;
    float lsum = 0.f;
    if (r.act) {
        wait_scores();   // of its own key block: the first group's exponentials run under the second block's products
        tc_fence_after();
        if (ok) lsum = request_probabilities(r, 0.f);
    }
    if (ROWS == 128 || row < ROWS) xs[g * ROWS + row] = lsum;
    const bool off_range = r.act && ok && counts && !(lsum > 0x1p-80f && lsum < 0x1p80f);
    if (named_bar_or(1, 256, off_range)) {
        // exact form: row maxima over both key blocks first
        float mx = -INFINITY;
        if (r.act && ok) {
#pragma unroll 1
            for (int c0 = 0; c0 < 128; c0 += 32) {
                uint32_t v[32];
                tmem_ld32(r.lane_base + (uint32_t)(g * 128 + c0), v);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    if (c0 + i < r.valid_cols) mx = fmaxf(mx, __uint_as_float(v[i]));
            }
        }
        if (ROWS == 128 || row < ROWS) xs[g * ROWS + row] = mx;
        named_bar_sync(1, 256);
        const float mt = fmaxf(mx, xs[(g ^ 1) * ROWS + (row & (ROWS - 1))]) * r.k2;   // an inactive group has published -inf
        named_bar_sync(1, 256);                                                        // both maxima are read: xs may now take the sums
        lsum = r.act && ok ? request_probabilities(r, mt) : 0.f;
        if (ROWS == 128 || row < ROWS) xs[g * ROWS + row] = lsum;
        named_bar_sync(1, 256);
    }
    return lsum + xs[(g ^ 1) * ROWS + (row & (ROWS - 1))];
}

// O times inv -> 64 columns of the first layer's input, bf16: dst is the row's 128 bytes of a 128B-swizzled K-major chunk (write: it has a place).
__device__ __forceinline__ void request_attention_row(const RequestRow &r, float inv, unsigned char *dst, bool write)
{
#pragma unroll 1
    for (int c0 = 0; c0 < 64; c0 += 32) {
        uint32_t v[32];
        tmem_ld32(r.lane_base + (uint32_t)(256 + 64 * r.g + c0), v);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(v[8 * q + 2 * i]) * inv, __uint_as_float(v[8 * q + 2 * i + 1]) * inv);
                w[i] = *reinterpret_cast<const uint32_t *>(&hh);
            }
            const int slot16 = (c0 >> 3) + q;
            if (write) *reinterpret_cast<uint4 *>(dst + ((slot16 ^ (r.row & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// Cross features (Section 3.3): the row of field f's user-side table that a candidate's bucket selects.
struct CrossTables {
    int32_t B, dc, b_mask, bucket_mode;   // b_mask: B - 1 where B is a power of two, else -1
};
// Eight columns from `col` on: their field, and where the field's tables begin for them (16-byte units).
struct CrossColumns {
    int f;
    uint32_t row16, base16;
};
__device__ __forceinline__ CrossColumns cross_columns(const CrossTables &c, int col)
{
    const int f = col / c.dc, kin = col - f * c.dc;
    const uint32_t row16 = (uint32_t)(c.dc >> 3);
    return CrossColumns{f, row16, (uint32_t)(f * c.B) * row16 + (uint32_t)(kin >> 3)};
}
__device__ __forceinline__ uint32_t cross_offset16(const CrossTables &c, const CrossColumns &at, int id)
{
    uint32_t bk;
    if (c.bucket_mode == AIF_BUCKET_MOD) bk = (uint32_t)(id % c.B);
    else {
        const uint64_t h = mix64((uint64_t)id, (uint64_t)at.f);
        bk = c.b_mask >= 0 ? (uint32_t)(h & (uint64_t)c.b_mask) : (uint32_t)(h % (uint64_t)c.B);
    }
    return bk * at.row16 + at.base16;
}

// The ids of a gather thread's rows r0, r0 + 16, ...: its warp has read every one once (lane l row 4 w + l % 4 + 16 (l / 4) of warp w's rows) and
// hands them round.  One outside the table becomes -1, whose rows are filled with zeros, and sets the status bit.
template <int N>
__device__ __forceinline__ void request_ids(int (&id)[N], int mine, int cnt, int64_t M, uint32_t *status, int lane, int sub, int r0)
{
#pragma unroll
    for (int i = 0; i < N; ++i) id[i] = __shfl_sync(0xffffffffu, mine, (lane >> 3) + 4 * i);
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (r0 + 16 * i < cnt && (id[i] < 0 || (int64_t)id[i] >= M)) {
            id[i] = -1;
            if (sub == 0) atomicOr(status, AIF_STATUS_BAD_ID);
        }
}

}  // namespace
}  // namespace aif
