// Scoring pass of a small request by clusters of four CTAs (sm_100a, bf16 storage), the same shapes as aif_tc_fused.cu.
//
// In the kernel of one CTA per tile every SM takes in all weights, 1.05 MB at 59 bytes per clock, and 1000 candidates are 8 tiles on 148 SMs:
// 37 k cycles whatever the machine could do beside.  Here a request's candidates go in tiles of 16 to 48, so many that all clusters of four find
// room at once, and the four CTAs of a cluster share the units: each forms 128 units of the first layer and a quarter of the
// second for all candidates of the tile, 260 KB of weights.  The layers' products are units x candidates (M = 128 units, N = the tile),
// so a narrow tile costs no padding.  Every CTA of a cluster gathers the tile's rows and does its attention (a few hundred keys for a few
// candidates: less than handing the rows round); the first layer's activations, 128 units of every candidate, go to the other three from
// shared memory to shared memory (8 KB each for 32 candidates), and the second layer's outputs to the first.
// Every sum is in the order of aif_tc_fused.cu (one accumulator over a layer's chunks and, last, its biases; the output layer's eight partial sums), so a
// candidate's logit is the same bits whichever kernel its call takes and whoever shares it.
// 1000 candidates, 200 behaviours: 20.2 us by the other kernel, 13.7 so; 200 candidates: 20.4 and 12.4; 1500: 20.5 and 15.8.
//
// Tried: products the other way round without sharing the units (a tile of 16 to 128 per CTA, all weights): 22.5 us for 1000 candidates, 41.5 for 10^4 with
// host buffers (37.0), three 32 KB stages of weights in flight being 43 bytes per clock; accumulators of its own for either issuing warp, which the
// epilogue adds (another order of sums): 13.9 for 1000; one issuing lane that asks for the next chunk's barrier ahead: 15.4; two chunks to a turn:
// 16.4, and 22 where the ring has three stages.
//
// Of 23 k cycles for 1000 candidates the set-up is 1.8 k, rows and scores 2.9 k, the softmax 3.3 k (a tile's rows lie in one or two warps'
// tensor-memory lanes), O and its rows 2.2 k, the layers 4.5 k and 3.8 k, their epilogues and the exchange 1.9 k, the CTAs' meeting 1.3 k, the
// output layer 1.5 k.
// 480 threads: warps 0-7 softmax and epilogues, 8 and 14 the issuers, 9-12 gather, 13 one lane of TMA, as there.  A chunk of 64 columns is four
// products of 45 cycles; the wait for its weights takes 140 cycles even where they are there, the hand-over between the issuers 180, the commit 100.
// Tensor memory: attention as there (scores [0, 256), O [256, 384), probabilities [384, 512)); then the layers' accumulators, D of the first at 0, of
// the second at 128.
// Every wait is bounded.
#include <cuda.h>

#include <mutex>

#include "aif_tc_request.cuh"

namespace aif {
namespace {

constexpr int kFThreads = 480;
constexpr int kFMmaWarp = 8, kFProdWarp0 = 9, kFBWarp = 13, kFMmaWarp2 = 14;
constexpr int kChunk = 16384;                  // 128 rows x 64 bf16
constexpr int kMaxCross = 8;                   // cross-feature chunks (64 columns each)
constexpr int kH1 = 512;
constexpr int kCtas = 4;                       // of a cluster
constexpr int kMaxTile = 48;
constexpr int kBStage = 16384, kMaxStages = 8;
constexpr int kMaxWeights = 4 + kMaxCross + kH1 / 64;   // chunks of weights of both layers, a barrier pair each
constexpr size_t kFSmem = 227 * 1024;
constexpr int kMiscBytes = 3072;               // barriers | row sums | output weights, flags
constexpr int kBias1 = 4096, kOnes = kMaxTile * 32, kBias = 2 * kBias1 + kOnes;   // bias operands: of either layer, and what they are multiplied by
// shared memory behind the miscellany, with c = tile x 128 bytes a chunk of 64 columns: E 2 c | key/value blocks 64 KB, later the attention
// chunks | cross chunks 8 c | activations 8 c | weight ring
constexpr int stages_for(int tile) { return ((int)kFSmem - 1024 - kMiscBytes - 65536 - 18 * tile * 128) / kBStage < kMaxStages ? ((int)kFSmem - 1024 - kMiscBytes - 65536 - 18 * tile * 128) / kBStage : kMaxStages; }
static_assert(stages_for(kMaxTile) >= 3, "weight ring");

enum {
    BAR_E_FULL = 0, BAR_KV_FULL, BAR_S_FULL = BAR_KV_FULL + 2, BAR_P_FULL = BAR_S_FULL + 2, BAR_O_FINAL, BAR_ATT_FULL, BAR_ACC1_FULL,
    BAR_H1_FULL, BAR_ACC2_FULL, BAR_TURN, BAR_FULL_A = BAR_TURN + 2, BAR_FULL_B = BAR_FULL_A + kMaxCross, BAR_EMPTY_B = BAR_FULL_B + kMaxWeights, BAR_COUNT = BAR_EMPTY_B + kMaxWeights
};
static_assert(BAR_COUNT * 8 + 16 <= 512, "barriers");
static_assert(2 * kMaxTile * 128 + kBias <= 32768, "attention rows and bias operands where the key blocks were");
// The second layer's outputs of all units, [candidate][row_floats], as the first CTA sums them up: in front of the activations.  Eight floats
// of padding, four of them in the middle: eight threads of a candidate and four candidates are on 32 banks.
__host__ __device__ constexpr int row_floats(int H2) { return H2 + 8; }
static_assert(kMaxTile * row_floats(256) * 4 <= 8 * kMaxTile * 128 + 32768 && 16 * row_floats(256) * 4 <= 8 * 16 * 128 + 32768, "second layer's outputs");
static_assert(kMaxTile * 8 <= kFThreads, "eight threads per candidate");

struct SplitParams {
    ScoreLaunch sl;
    const uint8_t *E;
    int64_t M;
    int32_t tile;           // candidates per cluster, a multiple of 16, at most kMaxTile
    int32_t stages;         // of the weight ring
    CrossTables cross;
    int32_t n_cross;
    int32_t H2, emit_sigmoid;
    float scale_log2;       // log2(e) / sqrt(d)
    const __nv_bfloat16 *b2_hl;   // [2][H2]: second-layer bias, high parts then remainders
    const __nv_bfloat16 *w_out;
    const float *b_out;
};

__global__ void __launch_bounds__(kFThreads, 1) k_request_split(const __grid_constant__ CUtensorMap tmapS,
                                                                const __grid_constant__ CUtensorMap tmapW1,
                                                                const __grid_constant__ CUtensorMap tmapW2, const SplitParams p)
{
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *misc = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(misc);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + BAR_COUNT);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    float *xs = reinterpret_cast<float *>(misc + 512);         // [2][64]: row sums or maxima of the two softmax groups
    float *wout_s = reinterpret_cast<float *>(misc + 1024);    // [H2] output weights
    float *ok_s = wout_s + 256;                                // [4]: all is well with a CTA (the first CTA's)
    uint32_t *good_s = reinterpret_cast<uint32_t *>(ok_s + 4); // [tile]: a candidate's id is in the table
    const int cs = p.tile * 128;
    unsigned char *smE = misc + kMiscBytes, *smKV = smE + 2 * cs, *smAtt = smKV, *smX = smKV + 65536, *smH = smX + 8 * cs, *smB = smH + 8 * cs;
    unsigned char *smBias1 = smAtt + 2 * cs, *smBias2 = smBias1 + kBias1, *smOnes = smBias2 + kBias1;
    float *smOut = reinterpret_cast<float *>(smH) - p.tile * row_floats(p.H2);
    auto bar = [&](int i) { return smem_u32(bars + i); };

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // (a role is a whole warp's, and the compiler sees it)
    const int rank = (int)cluster_rank(), cluster = (int)(blockIdx.x / kCtas);

    if (tid == 0) {
        mbar_init(bar(BAR_E_FULL), 128);
        mbar_init(bar(BAR_KV_FULL), 1);
        mbar_init(bar(BAR_KV_FULL + 1), 1);
        mbar_init(bar(BAR_S_FULL), 1);
        mbar_init(bar(BAR_S_FULL + 1), 1);
        mbar_init(bar(BAR_P_FULL), 256);
        mbar_init(bar(BAR_O_FINAL), 1);
        mbar_init(bar(BAR_ATT_FULL), 256);
        mbar_init(bar(BAR_ACC1_FULL), 2);
        mbar_init(bar(BAR_H1_FULL), 1);
        mbar_init(bar(BAR_ACC2_FULL), 2);
        mbar_init(bar(BAR_TURN), 1);
        mbar_init(bar(BAR_TURN + 1), 1);
        for (int i = 0; i < kMaxCross; ++i) mbar_init(bar(BAR_FULL_A + i), 128);
        for (int s = 0; s < kMaxWeights; ++s) mbar_init(bar(BAR_FULL_B + s), 1), mbar_init(bar(BAR_EMPTY_B + s), 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // The gather threads fetch their candidate ids while barriers and tensor memory are being set up: the ids head the
    // longest chain of dependent memory accesses of the kernel (ids -> item rows -> scores).
    int mine = -1;
    if (warp >= kFProdWarp0 && warp < kFBWarp) {
        grid_dep_wait();
        // (they may lie in host memory across the bus: a gather warp reads its rows' once and hands them round by shuffle, after the barrier)
        const int w = warp - kFProdWarp0, r = 4 * w + (lane & 3) + 16 * (lane >> 2);
        if (r < min(p.tile, p.sl.single.n - cluster * p.tile)) mine = p.sl.ids[p.sl.single.off + cluster * p.tile + r];
    }
    if (warp == kFMmaWarp) tmem_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // the other CTAs' barriers exist
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    grid_dep_launch();
    grid_dep_wait();

    const ReqDev rq = p.sl.single;
    const int start = cluster * p.tile, cnt = min(p.tile, rq.n - start);
    const int64_t pos0 = rq.off + start;
    const SlotDev *slot = p.sl.slots + rq.slot;
    const int L = slot->L;
    const int nb = L > 128 ? 2 : 1;
    const int n_k1 = 4 + p.n_cross;
    const float b_out = __ldg(p.b_out);   // (for the last step)

    if (warp < 8) {
        // ===================== softmax, epilogues =====================
        const int g = warp >> 2, wq = warp & 3, row = wq * 32 + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
        bool ok = true;
        // a wait of the whole warp: the tensor-memory loads and stores that follow need every lane to take the same branch
        auto wait = [&](int b) {
            const bool got = ok && mbar_wait(bar(b), 0u, abort_flag);
            ok = __all_sync(0xffffffffu, got);
        };
        bool good = false;
        if (row < cnt) {
            const int id = p.sl.ids[pos0 + row];
            good = id >= 0 && (int64_t)id < p.M;
        }
        if (g == 0 && row < p.tile) good_s[row] = good ? 1u : 0u;
        if (tid < p.H2) wout_s[tid] = __bfloat162float(p.w_out[tid]);
        // bias of this thread's unit, of the first layer (group 0: the request's cached user partial) or the second
        const int unit = rank * 128 + row, h2 = p.H2 / kCtas;
        const bool has2 = row < h2;
        uint32_t bias_hl = 0u;
        {
            const __nv_bfloat16 *hl = g == 0 ? reinterpret_cast<const __nv_bfloat16 *>(slot->pu_hl) : p.b2_hl;
            const int at = g == 0 ? unit : rank * h2 + row, n = g == 0 ? kH1 : p.H2;
            if (g == 0 || has2) bias_hl = (uint32_t)__bfloat16_as_ushort(hl[at]) | (uint32_t)__bfloat16_as_ushort(hl[n + at]) << 16;
        }
        // ---- attention: scores of key block g -> probabilities
        // (rows beyond the tile: nobody's; the products read whatever lies there)
        const RequestRow rr{lane_base, g, row, L - g * 128 < 128 ? L - g * 128 : 128, g < nb && wq * 32 < p.tile, p.scale_log2};
        const float l_all = request_softmax<64>(rr, xs, ok, row < p.tile, [&] { wait(BAR_S_FULL + g); });
        tc_fence_before();
        mbar_arrive(bar(BAR_P_FULL));
        // ---- O -> attention chunk g of the first layer's input (64 columns, 128B-swizzled K-major)
        wait(BAR_O_FINAL);
        tc_fence_after();
        if (ok && wq * 32 < p.tile) request_attention_row(rr, good ? 1.0f / l_all : 0.f, smAtt + g * cs + row * 128, row < p.tile);
        // The biases are added by the tensor cores, as in aif_tc_fused.cu: one more step of K = 16 whose operands are, per unit, the bias in two
        // bf16 values (high part, remainder) and, per candidate, two ones (no swizzle: 16-byte columns, the second ones zero).
        if (ok) {
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            uint4 *b = reinterpret_cast<uint4 *>(g == 0 ? smBias1 : smBias2);
            b[row] = make_uint4(bias_hl, 0u, 0u, 0u), b[128 + row] = zero;
            if (g == 0 && row < p.tile) {
                uint4 *one = reinterpret_cast<uint4 *>(smOnes);
                one[row] = make_uint4(0x3F803F80u, 0u, 0u, 0u), one[p.tile + row] = zero;
            }
        }
        fence_proxy_async();   // the MMA reads these chunks through the async proxy
        tc_fence_before();
        mbar_arrive(bar(BAR_ATT_FULL));
        // ---- layer-1 epilogue: a thread owns a unit (lane) and, with the other group, every second sixteen candidates (columns).  ReLU, bf16, and
        // the activations go to shared memory as the second layer's operand: 64-unit chunks of 128-byte rows, one per candidate; this
        // CTA's two chunks then go to the other three.
        wait(BAR_ACC1_FULL);
        tc_fence_after();
        if (ok) {
            unsigned char *dst = smH + (unit >> 6) * cs + (unit & 7) * 2;
            const int piece = (unit & 63) >> 3;
#pragma unroll 1
            for (int c0 = 16 * g; c0 < p.tile; c0 += 32) {
                uint32_t r[16];
                tmem_ld16(lane_base + (uint32_t)c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    *reinterpret_cast<__nv_bfloat16 *>(dst + (c0 + c) * 128 + ((piece ^ (c & 7)) << 4)) = __float2bfloat16_rn(fmaxf(__uint_as_float(r[c]), 0.f));
            }
        }
        fence_proxy_async();   // read by the copies and the MMA through the async proxy
        tc_fence_before();
        if (!named_bar_or(1, 256, !ok) && tid == 0) {
            mbar_expect_tx(bar(BAR_H1_FULL), (uint32_t)((kCtas - 1) * 2 * cs));
            const uint32_t src = smem_u32(smH + 2 * rank * cs);
            for (int q = 1; q < kCtas; ++q) {
                const uint32_t to = (uint32_t)((rank + q) % kCtas);
                bulk_copy_cluster(cluster_addr(src, to), src, (uint32_t)(2 * cs), cluster_addr(bar(BAR_H1_FULL), to));
            }
        }
        // ---- layer-2 epilogue: unit (lane) of this CTA's quarter, ReLU, into the first CTA's shared memory
        wait(BAR_ACC2_FULL);
        tc_fence_after();
        if (ok && wq * 32 < h2) {
            const int unit2 = rank * h2 + row, stride = row_floats(p.H2);
            const uint32_t out = cluster_addr(smem_u32(smOut + unit2 + (unit2 >= p.H2 / 2 ? 4 : 0)), 0u);
#pragma unroll 1
            for (int c0 = 16 * g; c0 < p.tile; c0 += 32) {
                uint32_t r[16];
                tmem_ld16(lane_base + 128u + (uint32_t)c0, r);
                tmem_ld_wait();
                if (has2)
#pragma unroll
                    for (int c = 0; c < 16; ++c) st_cluster_f32(out + (uint32_t)((c0 + c) * stride * 4), fmaxf(__uint_as_float(r[c]), 0.f));
            }
        }
        const bool all_ok = !named_bar_or(1, 256, !ok);   // a wait that ran out anywhere in these warps
        if (tid == 0) st_cluster_f32(cluster_addr(smem_u32(ok_s + rank), 0u), all_ok ? 1.f : 0.f);
    } else if (warp == kFMmaWarp || warp == kFMmaWarp2) {
        // ===================== MMA issuers: even and odd chunks of the layers; the attention is the first one's =====================
        // The whole warp walks through, one lane issues.  (With the walk in one lane, behind a branch, its descriptors are no uniform values
        // to the compiler and a product takes 75 cycles to issue: 15.9 us for 1000 candidates.)
        const bool one = elect_one();
        constexpr uint32_t idesc_qk = umma_idesc_bf16(kTcTile, 128);
        constexpr uint32_t idesc_pv = umma_idesc_bf16_bmn(kTcTile, 128);
        const uint32_t idesc_l = umma_idesc_bf16(128, p.tile);   // of both layers: 128 units x the tile's candidates
        const int second = warp == kFMmaWarp2;
        bool ok = mbar_wait(bar(BAR_E_FULL), 0u, abort_flag);
        fence_proxy_async();   // the item rows were written by cp.async
        if (!second) {
            // scores = Q K^T, one key block after the other
            const uint64_t qd = umma_desc_sw128(smem_u32(smE));
            for (int j = 0; ok && j < nb; ++j) {
                ok = mbar_wait(bar(BAR_KV_FULL + j), 0u, abort_flag);
                tc_fence_after();
                if (!ok) break;
                const uint64_t kd = umma_desc_sw128(smem_u32(smKV + j * 32768));
                const uint32_t d_tmem = tmem_base + (uint32_t)(j * 128);
                if (one) {
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        umma_bf16(d_tmem, qd + (uint64_t)(uint32_t)((kk >> 2) * (cs >> 4) + 2 * (kk & 3)), kd + (uint64_t)((kk >> 2) * (kChunk >> 4) + 2 * (kk & 3)), idesc_qk, kk > 0 ? 1u : 0u);
                    umma_commit(bar(BAR_S_FULL + j));
                }
            }
            // O = P V: the probabilities from tensor memory, V = the key blocks read MN-major
            ok = ok && mbar_wait(bar(BAR_P_FULL), 0u, abort_flag);
            tc_fence_after();
            if (ok && one) {
                for (int j = 0; j < nb; ++j) {
                    const uint64_t vd = umma_desc_mn_sw128(smem_u32(smKV + j * 32768), kChunk);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        umma_bf16_ts(tmem_base + 256u, tmem_base + (uint32_t)(384 + j * 64 + kk * 8), vd + (uint64_t)(kk * (2048 >> 4)), idesc_pv,
                                     (j > 0 || kk > 0) ? 1u : 0u);
                }
                umma_commit(bar(BAR_O_FINAL));
            }
        }
        // The chunks of a layer in their order, then its biases, into one accumulator: a candidate's sums are those of the kernel of one CTA per
        // tile, bit for bit.  The two warps take turns, so the order of their products is that of the hand-overs between them; what comes
        // before a chunk's products (waits, descriptors) and behind them (commits) is in nobody's way.
        ok = ok && mbar_wait(bar(BAR_ATT_FULL), 0u, abort_flag);
        tc_fence_after();
        uint32_t turn = 0;   // of this warp: every second chunk of both layers
        int sb = second % p.stages;
        auto product = [&](int c, uint32_t d_tmem, uint64_t xd, bool first, const unsigned char *bias) {   // weight chunk c, of both layers in their order
            if (!(ok = mbar_wait(bar(BAR_FULL_B + c), 0u, abort_flag))) return;
            tc_fence_after();
            const uint64_t wd = umma_desc_sw128(smem_u32(smB + sb * kBStage));
            if (c > 0 && !(ok = mbar_wait(bar(BAR_TURN + second), (turn - (uint32_t)!second) & 1u, abort_flag))) return;
            ++turn;
            tc_fence_after();
            if (one) {
                umma_bf16(d_tmem, wd, xd, idesc_l, first ? 0u : 1u);
#pragma unroll
                for (int kk = 1; kk < 4; ++kk) umma_bf16_acc(d_tmem, wd + (uint64_t)(2 * kk), xd + (uint64_t)(2 * kk), idesc_l);
                if (bias) umma_bf16_acc(d_tmem, umma_desc_plain(smem_u32(bias), 2048), umma_desc_plain(smem_u32(smOnes), (uint32_t)p.tile * 16u), idesc_l);
                tc_fence_before();
                mbar_arrive(bar(BAR_TURN + (second ^ 1)));
                umma_commit(bar(BAR_EMPTY_B + c));
            }
            for (sb += 2; sb >= p.stages;) sb -= p.stages;
        };
        // layer 1: K chunks [ item 0-1 | attention 2-3 | cross 4.. ], this CTA's 128 units
        int c = second;
        for (; ok && c < n_k1; c += 2) {
            if (c >= 4) {
                if (!(ok = mbar_wait(bar(BAR_FULL_A + c - 4), 0u, abort_flag))) break;
                fence_proxy_async();
            }
            product(c, tmem_base, umma_desc_sw128(smem_u32(c < 2 ? smE + c * cs : c < 4 ? smAtt + (c - 2) * cs : smX + (c - 4) * cs)), c == 0, c == n_k1 - 1 ? smBias1 : nullptr);
        }
        if (ok && one) umma_commit(bar(BAR_ACC1_FULL));
        // layer 2, this CTA's quarter of the units (lanes beyond it: whatever the stage held, nobody reads them)
        ok = ok && mbar_wait(bar(BAR_H1_FULL), 0u, abort_flag);
        tc_fence_after();
        for (; ok && c < n_k1 + kH1 / 64; c += 2)
            product(c, tmem_base + 128u, umma_desc_sw128(smem_u32(smH + (c - n_k1) * cs)), c == n_k1, c == n_k1 + kH1 / 64 - 1 ? smBias2 : nullptr);
        if (ok && one) umma_commit(bar(BAR_ACC2_FULL));
        __syncwarp();
    } else if (warp < kFBWarp) {
        // ===================== item-row and cross-feature gather (128 threads) =====================
        const int pt = tid - kFProdWarp0 * 32;
        const int sub = pt & 7, r0 = pt >> 3;   // 16-byte slot of the 128-byte chunk row; rows r0, r0 + 16, r0 + 32
        constexpr int kR = kMaxTile / 16;
        const uint32_t row_off = (uint32_t)(r0 * 128) + (uint32_t)((sub ^ (r0 & 7)) << 4);
        int id[kR];
        request_ids(id, mine, cnt, p.M, p.sl.status, lane, sub, r0);
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            if (16 * i >= p.tile) break;
            const uint8_t *gsrc = p.E + (id[i] >= 0 ? (size_t)id[i] * 256 + sub * 16 : 0);
            const uint32_t dst = smem_u32(smE) + row_off + (uint32_t)(i * 16 * 128);
            cp_async16(dst, gsrc, id[i] >= 0 ? 16u : 0u);
            cp_async16(dst + (uint32_t)cs, gsrc + 128, id[i] >= 0 ? 16u : 0u);
        }
        cp_async_arrive_noinc(bar(BAR_E_FULL));
        // cross features (Section 3.3): the row of field f's user-side table that the candidate's bucket selects
        const uint8_t *Tt = reinterpret_cast<const uint8_t *>(slot->T);
        for (int n = 0; n < p.n_cross; ++n) {
            const CrossColumns at = cross_columns(p.cross, 64 * n + 8 * sub);
            const uint32_t dst0 = smem_u32(smX + n * cs) + row_off;
#pragma unroll
            for (int i = 0; i < kR; ++i) {
                if (16 * i >= p.tile) break;
                const uint32_t off = cross_offset16(p.cross, at, id[i]);
                cp_async16(dst0 + (uint32_t)(i * 16 * 128), id[i] >= 0 ? Tt + ((size_t)off << 4) : p.E, id[i] >= 0 ? 16u : 0u);
            }
            cp_async_arrive_noinc(bar(BAR_FULL_A + n));
        }
        cp_async_wait_all();
    } else {
        // ===================== key/value blocks and weights (TMA) =====================
        if (lane == 0) {
            for (int j = 0; j < nb; ++j) {
                mbar_expect_tx(bar(BAR_KV_FULL + j), 32768u);
                tma_load_3d(smem_u32(smKV + j * 32768), &tmapS, bar(BAR_KV_FULL + j), 0, j * 128, rq.slot);
                tma_load_3d(smem_u32(smKV + j * 32768 + kChunk), &tmapS, bar(BAR_KV_FULL + j), 64, j * 128, rq.slot);
            }
            int sb = 0;
            for (int kc = 0; kc < n_k1 + kH1 / 64; ++kc) {
                if (kc >= p.stages && !mbar_wait(bar(BAR_EMPTY_B + kc - p.stages), 0u, abort_flag)) break;
                const bool first = kc < n_k1;
                mbar_expect_tx(bar(BAR_FULL_B + kc), first ? 16384u : (uint32_t)(p.H2 / kCtas) * 128u);
                if (first) tma_load_2d(smem_u32(smB + sb * kBStage), &tmapW1, bar(BAR_FULL_B + kc), kc * 64, rank * 128);
                else tma_load_2d(smem_u32(smB + sb * kBStage), &tmapW2, bar(BAR_FULL_B + kc), (kc - n_k1) * 64, rank * (p.H2 / kCtas));
                if (++sb == p.stages) sb = 0;
            }
        }
        __syncwarp();
    }

    // ---- teardown: everybody arrives here, also after an abort
    if (*abort_flag) {
        if (tid == 0) atomicOr(p.sl.status, AIF_STATUS_TIMEOUT);
        // let copies and MMAs that are still in flight land before shared memory and TMEM go away
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // all partial logits are with the first CTA; nobody leaves while another may still write to it
    if (rank == 0) {
        // The output layer, in the order of the kernel of one CTA per tile: eight threads per candidate, each every fourth unit of one half
        const int cand = tid >> 3, half = (tid >> 2) & 1, i = tid & 3, hn = p.H2 / 2;
        float dot = 0.f;
        if (cand < cnt) {
            const float *v = smOut + cand * row_floats(p.H2) + half * (hn + 4) + i, *w = wout_s + half * hn + i;
#pragma unroll 16
            for (int k = 0; k < hn; k += 4) dot = fmaf(v[k], w[k], dot);
        }
        dot += __shfl_xor_sync(0xffffffffu, dot, 1);
        dot += __shfl_xor_sync(0xffffffffu, dot, 2);
        dot += __shfl_xor_sync(0xffffffffu, dot, 4);
        if (cand < cnt && (tid & 7) == 0) {
            float logit = dot + b_out;
            const bool all = ok_s[0] != 0.f && ok_s[1] != 0.f && ok_s[2] != 0.f && ok_s[3] != 0.f;
            if (p.emit_sigmoid) logit = 1.0f / (1.0f + expf(-logit));
            p.sl.logits[pos0 + cand] = good_s[cand] && all ? logit : __int_as_float(0x7fc00000);   // no number for a bad id, nor where a wait ran out
        }
    }
    if (warp == kFMmaWarp) tmem_dealloc(tmem_base, 512);
}

}  // namespace

// Clusters of four that the machine holds at once (0: not usable).
int tc_split_prepare()
{
    if (cudaFuncSetAttribute(k_request_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFSmem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kCtas), cfg.blockDim = dim3(kFThreads), cfg.dynamicSmemBytes = kFSmem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kCtas, attr.val.clusterDim.y = 1, attr.val.clusterDim.z = 1;
    cfg.attrs = &attr, cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_request_split, &cfg) != cudaSuccess) cudaGetLastError(), n = 0;
    return n;
}

// The streams of a device's last small requests, of all contexts: how many of them run beside each other as far as a call can know.  A hint
// that decides on speed alone; a handle is compared, never used.
struct RecentStreams {
    static constexpr int kCalls = 8;
    std::mutex lock;
    cudaStream_t stream[kCalls];
    int calls = 0;
    int note(cudaStream_t st)   // different streams among the last calls, this one included
    {
        const std::lock_guard<std::mutex> guard(lock);
        stream[calls++ % kCalls] = st;
        if (calls == 2 * kCalls) calls = kCalls;
        int different = 0;
        for (int i = 0, n = calls < kCalls ? calls : kCalls; i < n; ++i) {
            bool seen = false;
            for (int j = 0; j < i; ++j) seen = seen || stream[j] == stream[i];
            different += !seen;
        }
        return different;
    }
};
static RecentStreams g_recent[16];

// Candidates per cluster for a single request of n, 0: the kernel of one CTA per tile is the better one (the caller has checked tc_fused_supported
// and the sequence's length).  Clusters make a call shorter by taking more of the machine: 1000 candidates hold 128 SMs for 14 us in place of 8
// for 20.  So they are taken where as many calls as there are streams at work are one round of clusters together.  1000 candidates on
// 1, 2, 4 and 8 streams, us per call: clusters 13.5, 12.2, 12.1, 12.1, one CTA per tile 20.1, 10.4, 5.4, 2.9; 200 candidates 12.0, 6.3, 4.8, 4.7
// and 20.4, 10.3, 5.3, 2.8.
int tc_split_tile(const aif_ctx *ctx, int n, cudaStream_t st)
{
    if (n > ctx->split_clusters * kMaxTile) return 0;
    const int calls = ctx->device < 16 ? g_recent[ctx->device].note(st) : 1;
    for (int tile = 16; tile <= kMaxTile; tile += 16)
        if ((n + tile - 1) / tile * calls <= ctx->split_clusters) return tile;
    return 0;
}

cudaError_t launch_request_split(const aif_ctx *ctx, const ScoreLaunch &sl, int tile, cudaStream_t st)
{
    const aif_config &c = ctx->cfg;
    SplitParams p{};
    p.sl = sl, p.E = (const uint8_t *)ctx->E, p.M = c.M;
    p.tile = tile, p.stages = stages_for(tile);
    p.cross = CrossTables{c.B, c.dc, (c.B & (c.B - 1)) == 0 ? c.B - 1 : -1, c.bucket_mode};
    p.n_cross = c.F * c.dc / 64;
    p.H2 = c.hidden[1], p.emit_sigmoid = c.emit_sigmoid;
    p.scale_log2 = 1.4426950408889634f / sqrtf((float)c.d);
    p.b2_hl = reinterpret_cast<const __nv_bfloat16 *>(ctx->tc_fused_plan), p.w_out = (const __nv_bfloat16 *)ctx->w_out, p.b_out = ctx->b_out;
    const CUtensorMap *ms = reinterpret_cast<const CUtensorMap *>(tc_att_tmap(ctx));
    const CUtensorMap *m1 = reinterpret_cast<const CUtensorMap *>(tc_weight_half_tmap(ctx, 0));
    const CUtensorMap *m2 = reinterpret_cast<const CUtensorMap *>(tc_weight_quarter_tmap(ctx));
    const int grid = (sl.single.n + p.tile - 1) / p.tile * kCtas;
    cudaError_t e = launch_pdl_cluster(k_request_split, dim3(grid), dim3(kFThreads), kFSmem, kCtas, st, *ms, *m1, *m2, p);
    count_launch();
    return e;
}

}  // namespace aif
