// What follows the attention in a block, in one kernel, for d_model = 256 and many rows:
//     mid = x + att Wo^T + bo,   x <- mid + W2 SiLU(W1 LN(mid; g, b) + b1) + b2
// Persistent CTA pairs (a cluster of two, tcgen05 cta_group::2), 256 rows of the residual stream per pair and tile, 128 per CTA.
// Per tile, in each CTA's TMEM and shared memory:
//     att Wo^T                attention rows (A) and half of Wo's rows (B) by TMA; fp32 in the columns of the two S buffers
//     O = mid = x + att Wo^T + bo     eight warps, half a row per thread; mid into O's columns, LN(mid) as bf16 into the tile the
//                             attention rows came in
//     per 128 hidden units:   S = LN(mid) W1c^T (fp32, double-buffered), H = SiLU(S + b1c) (bf16, over S's own columns),
//                             O += H W2c^T (A from TMEM)
//     x  = O + b2             drained through shared memory as bulk tensor stores
//
// Why pairs.  A single CTA moves 320 KB through shared memory per chunk (both MMAs' operands, both weight tiles written by TMA):
// 2500 clocks at 128 B / clk where the MMAs need 2048.  In a pair each CTA holds half of every weight tile: 192 KB, and the
// MMAs set the pace.  The halved weight ring also makes room for a 64 KB staging area, so that x travels without stopping the
// tensor pipe: the next tile's rows arrive in two halves during the chunk loop and wait in registers, and a
// tile is drained while the next one's projection runs.  (Row-per-thread loads of x straight from global memory were
// measured: 9400 clocks per tile, 32 different lines per instruction.)  What stays serial per tile is drain -> LayerNorm ->
// first S and SiLU.
// With x added into O before the feed-forward products, the drain stores x instead of add-reducing into it: an fp32 reduction
// in L2 costs about twice a store (23 B / clk per SM with all SMs draining).
//
// Warp roles (384 threads): warp 0 = weight producer (and attention rows), warp 1 = TMEM owner + MMA issuer (the even CTA's
// issues for both), warp 2 = x producer, warp 3 none, warps 4-11 = LayerNorm, SiLU, drain (two warps per TMEM quadrant, each
// with half of the columns).  TMEM: O 0..255, S buffers 256..383 and 384..511.  The MMA warp issues S(0), S(1), then per chunk
// O += H(c) W2c^T, S(c+2): the tensor pipe executes in issue order, so S(c+2) cannot overwrite the buffer H(c) sits in before it
// has been consumed.  Chunks are counted over the CTA's whole life; buffers and barrier phases follow from that count.
#include "ffn_common.cuh"
#include "kernels.cuh"

namespace relaygr {

namespace {

using namespace ffn;

constexpr int kEpiRegs = 224, kOtherRegs = 56;       // registers per thread after the split: of the epilogue warps, of the other four
constexpr int kStageBytes = 16 * 1024, kStages = 5;  // a stage: this CTA's half of a K block of Wo, of half a W1 chunk, of half a W2 chunk
constexpr int kPatch = 4096;                         // 32 rows x 32 fp32 columns
constexpr int kOffW = kABytes;
constexpr int kOffStg = kOffW + kStages * kStageBytes;          // two patches per epilogue warp
constexpr int kOffB1 = kOffStg + 2 * kEpiWarps * kPatch;
constexpr int kOffB2 = kOffB1 + kMaxF * 4;
constexpr int kOffG = kOffB2 + kD * 4;               // LayerNorm gain and offset, out-proj bias: 3 x 256 floats
constexpr int kOffStat = kOffG + 3 * kD * 4;         // statistics of half rows: 2 x 128 pairs
constexpr int kOffBars = kOffStat + 2 * kRows * 8;
constexpr int kSmemBytes = kOffBars + 256 + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");

// [L]: the even CTA's copy counts for the pair
struct Bars {
    uint64_t w_full[kStages], w_empty[kStages];      // [L] / each CTA's own (committed to both)
    uint64_t att_full, a_ready, h_full[2];           // [L] attention rows landed / LN(mid) in shared memory / H in TMEM
    uint64_t o1_full, s_full[2], o_full;             // committed to both: projection, S, O complete
    uint64_t x_full[2], stg_free;                    // own: half of x landed / the staging area may be filled again
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(sizeof(Bars) <= 256, "barrier block");

template <int V> struct Int { static constexpr int value = V; };

__global__ void __launch_bounds__(kThreads, 1)
ffn_pair_kernel(const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmX,
                const __grid_constant__ CUtensorMap tmAtt, const __grid_constant__ CUtensorMap tmWo, const float *__restrict__ x,
                const float *__restrict__ g, const float *__restrict__ b, const float *__restrict__ b1, const float *__restrict__ b2,
                const float *__restrict__ bo, int64_t M, int F, float eps, int *err)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = smem, *sW = smem + kOffW, *stg = smem + kOffStg;
    float *b1s = reinterpret_cast<float *>(smem + kOffB1), *b2s = reinterpret_cast<float *>(smem + kOffB2);
    float *gs = reinterpret_cast<float *>(smem + kOffG), *bs = gs + kD, *bos = bs + kD;
    float2 *stat = reinterpret_cast<float2 *>(smem + kOffStat);
    Bars *bars = reinterpret_cast<Bars *>(smem + kOffBars);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)tc::cluster_ctarank();
    const bool leader = rank == 0;
    const int tile0 = blockIdx.x / 2, tile_step = gridDim.x / 2, n_tiles = (int)((M + 2 * kRows - 1) / (2 * kRows));
    const int nc = F / kChunk;
    auto row0_of = [&](int tile) { return tile * (2 * kRows) + rank * kRows; };
    // a stage of the ring: this CTA's share, counted (both shares) on the even CTA's barrier
    auto stage_expect = [&](int s) { if (leader) tc::mbar_expect_tx(&bars->w_full[s], 2 * kStageBytes); return tc::cluster_addr(&bars->w_full[s], 0); };
    auto load_wo = [&](int s, int kb) { tc::tma_load_2d_pair(sW + s * kStageBytes, &tmWo, kb * 64, rank * 128, stage_expect(s)); };

    // set-up that touches nothing earlier kernels wrote
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { tc::mbar_init(&bars->w_full[s], 1); tc::mbar_init(&bars->w_empty[s], 1); }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&bars->s_full[i], 1); tc::mbar_init(&bars->h_full[i], 2 * kEpiWarps);
            tc::mbar_init(&bars->x_full[i], 1);
        }
        tc::mbar_init(&bars->stg_free, kEpiWarps);
        tc::mbar_init(&bars->att_full, 1); tc::mbar_init(&bars->o1_full, 1); tc::mbar_init(&bars->o_full, 1);
        tc::mbar_init(&bars->a_ready, 2 * kEpiWarps);
        tc::fence_mbar_init();
        tc::tma_prefetch_desc(&tmW1); tc::tma_prefetch_desc(&tmW2); tc::tma_prefetch_desc(&tmX); tc::tma_prefetch_desc(&tmAtt); tc::tma_prefetch_desc(&tmWo);
    }
    if (warp == 1) {
        tc::tmem_alloc_pair(&bars->tmem_slot, kTmemCols);
        tc::tmem_relinquish_pair();
    }
    if (warp >= 4) {
        for (int i = threadIdx.x - 128; i < F; i += kEpiThreads) b1s[i] = b1 ? 0.5f * b1[i] : 0.f;      // SiLU takes half of its argument
        for (int i = threadIdx.x - 128; i < kD; i += kEpiThreads) {
            b2s[i] = b2 ? b2[i] : 0.f;
            gs[i] = g[i]; bs[i] = b[i]; bos[i] = bo ? bo[i] : 0.f;
        }
    }
    tc::cluster_sync();                               // the peer's barriers exist before anything signals them
    if (threadIdx.x == 0)
        for (int kb = 0; kb < 4; ++kb) load_wo(kb, kb);      // parameters, as the biases above
    grid_launch_dependents();
    grid_dependency_wait();                           // from here on: data of earlier kernels
    if (threadIdx.x == 0) bars->abort_flag = *reinterpret_cast<volatile int *>(err);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem_base = bars->tmem_slot;
    const bool live = bars->abort_flag == 0;

    // The epilogue keeps half a row of x (128 values) beside its working set.  Each warpgroup executes its instruction as a whole;
    // the two sizes add up to what the block was launched with (checked before the first launch), so the increase cannot wait for ever.
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
        if (!live) {
            if (threadIdx.x == 0 && leader)           // what was requested above lands before the pair ends
                for (int s = 0; s < 4; ++s) tc::mbar_wait(&bars->w_full[s], 0, err);
        } else if (warp == 0) {
            // ------------------------------------------------------------ weights, in the order of consumption: Wo in four K blocks,
            // W1(0), W1(1), then per chunk c: W2(c), W1(c+2); and the attention rows
            if (lane == 0) {
                int next = 4, phase = 0;              // of the ring; the first tile's Wo is on its way
                bool ok = true;
                auto acquire = [&] {
                    const int s = next;
                    ok = ok && tc::mbar_wait(&bars->w_empty[s], phase ^ 1, err);
                    if (++next == kStages) { next = 0; phase ^= 1; }
                    return s;
                };
                auto load = [&](bool second, int c) {
                    for (int half = 0; half < 2; ++half) {
                        const int s = acquire();
                        if (!ok) return;
                        uint8_t *dst = sW + s * kStageBytes;
                        const uint32_t bar = stage_expect(s);
                        if (!second) {                // 64 of the chunk's 128 rows of W1 [F, 256], K blocks 2*half and 2*half + 1
                            tc::tma_load_2d_pair(dst, &tmW1, (2 * half) * 64, c * kChunk + rank * 64, bar);
                            tc::tma_load_2d_pair(dst + kStageBytes / 2, &tmW1, (2 * half + 1) * 64, c * kChunk + rank * 64, bar);
                        } else {                      // 128 of the 256 rows of W2 [256, F], 64 hidden columns
                            tc::tma_load_2d_pair(dst, &tmW2, c * kChunk + half * 64, rank * 128, bar);
                        }
                    }
                };
                auto load_att = [&](int tile) {
                    if (leader) tc::mbar_expect_tx(&bars->att_full, 2 * kABytes);
                    const uint32_t bar = tc::cluster_addr(&bars->att_full, 0);
                    for (int kb = 0; kb < 4; ++kb) tc::tma_load_2d_pair(sA + kb * kKBlock, &tmAtt, kb * 64, row0_of(tile), bar);
                };
                load_att(tile0);
                int gc = 0;                           // chunks so far
                for (int tile = tile0; tile < n_tiles && ok; tile += tile_step) {
                    if (gc > 0) {
                        // the last S of the tile before has read A
                        ok = tc::mbar_wait(&bars->s_full[(gc - 1) & 1], ((gc - 1) >> 1) & 1, err);
                        if (ok) load_att(tile);
                        for (int kb = 0; kb < 4 && ok; ++kb) {
                            const int s = acquire();
                            if (ok) load_wo(s, kb);
                        }
                    }
                    for (int c = 0; c < 2 && c < nc && ok; ++c) load(false, c);
                    for (int c = 0; c < nc && ok; ++c) {
                        load(true, c);
                        if (c + 2 < nc && ok) load(false, c + 2);
                    }
                    gc += nc;
                }
            }
        } else if (warp == 1 && leader) {
            // ------------------------------------------------------------ MMA issuer (convergent warp, one elected lane issues)
            constexpr uint32_t idesc_s = tc::make_idesc(2 * kRows, kChunk, 0, 0);      // A and W1 both K-major
            constexpr uint32_t idesc_o = tc::make_idesc(2 * kRows, kD, 0, 0);          // att (or H from TMEM), Wo / W2 K-major
            const uint32_t a0 = tc::smem_u32(sA);
            int next = 0, phase = 0;                  // of the ring
            int gc = 0;
            bool ok = true;
            auto stage = [&] {                        // the next stage, complete in both CTAs
                const int s = next;
                ok = tc::mbar_wait(&bars->w_full[s], phase, err);
                tc::tc_fence_after();
                if (++next == kStages) { next = 0; phase ^= 1; }
                return s;
            };
            for (int tile = tile0, n = 0; tile < n_tiles && ok; tile += tile_step, ++n) {
                ok = tc::mbar_wait(&bars->att_full, n & 1, err);
                for (int kb = 0; kb < 4 && ok; ++kb) {          // att Wo^T, in the columns of both S buffers: the last H has been consumed by then
                    const int s = stage();
                    if (!ok) break;
                    const uint64_t adesc = tc::smem_desc_sw128(a0 + kb * kKBlock), bdesc = tc::smem_desc_sw128(tc::smem_u32(sW + s * kStageBytes));
                    if (tc::elect_one()) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) tc::mma_ss_pair(tmem_base + kColS, adesc + 2 * k, bdesc + 2 * k, idesc_o, (kb | k) != 0);
                        tc::mma_commit_pair(&bars->w_empty[s], 3);
                        if (kb == 3) tc::mma_commit_pair(&bars->o1_full, 3);
                    }
                    __syncwarp();
                }
                if (ok) ok = tc::mbar_wait(&bars->a_ready, n & 1, err);
                auto issue_s = [&](int c) {           // S = LN(mid) W1c^T
                    const int buf = (gc + c) & 1;
                    for (int half = 0; half < 2 && ok; ++half) {
                        const int s = stage();
                        if (!ok) break;
                        const uint32_t w = tc::smem_u32(sW + s * kStageBytes);
                        if (tc::elect_one()) {
#pragma unroll
                            for (int kb = 0; kb < 2; ++kb) {
                                const uint64_t adesc = tc::smem_desc_sw128(a0 + (2 * half + kb) * kKBlock), bdesc = tc::smem_desc_sw128(w + kb * (kStageBytes / 2));
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    tc::mma_ss_pair(tmem_base + kColS + buf * kChunk, adesc + 2 * k, bdesc + 2 * k, idesc_s, (half | kb | k) != 0);
                            }
                            tc::mma_commit_pair(&bars->w_empty[s], 3);
                            if (half == 1) tc::mma_commit_pair(&bars->s_full[buf], 3);
                        }
                        __syncwarp();
                    }
                };
                auto issue_o = [&](int c) {           // O += H W2c^T
                    const uint32_t hcol = kColS + ((gc + c) & 1) * kChunk;
                    for (int half = 0; half < 2 && ok; ++half) {
                        const int s = stage();
                        if (!ok) break;
                        const uint64_t bdesc = tc::smem_desc_sw128(tc::smem_u32(sW + s * kStageBytes));
                        if (tc::elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k)      // 16 hidden units per instruction: 8 TMEM columns of H, 32 bytes of every W2 row
                                tc::mma_ts_pair(tmem_base + kColO, tmem_base + hcol + half * 64 + k * 8, bdesc + 2 * k, idesc_o, 1);
                            tc::mma_commit_pair(&bars->w_empty[s], 3);
                            if (half == 1 && c == nc - 1) tc::mma_commit_pair(&bars->o_full, 3);
                        }
                        __syncwarp();
                    }
                };
                if (ok) issue_s(0);
                if (ok && nc > 1) issue_s(1);
                for (int c = 0; c < nc && ok; ++c) {
                    ok = tc::mbar_wait(&bars->h_full[(gc + c) & 1], ((gc + c) >> 1) & 1, err);      // H is in TMEM (and S in registers)
                    if (!ok) break;
                    issue_o(c);
                    if (ok && c + 2 < nc) issue_s(c + 2);
                }
                gc += nc;
            }
        } else if (warp == 2 && lane == 0) {
            // ------------------------------------------------------------ x, two halves per tile: of each epilogue warp's four
            // patches (32 rows x 32 columns) the first two, then the last two (of the first tile only the first: nothing has been
            // computed yet, so the epilogue fetches the rest itself at the same time).  What frees the staging area for load k + 1, in
            // order: first half of tile 0 in registers; then per tile: first half of the next in registers, tile drained.
            int k = 0;
            bool ok = true;
            for (int tile = tile0, n = 0; tile < n_tiles && ok; tile += tile_step, ++n)
                for (int h = 0; h < (n == 0 ? 1 : 2) && ok; ++h, ++k) {
                    if (k > 0) ok = tc::mbar_wait(&bars->stg_free, (k - 1) & 1, err);
                    if (!ok) break;
                    tc::mbar_expect_tx(&bars->x_full[h], 2 * kEpiWarps * kPatch);
                    for (int p = 0; p < 2 * kEpiWarps; ++p) {
                        const int ew = p >> 1, col = (ew >> 2) * 128 + (2 * h + (p & 1)) * 32;
                        tc::tma_load_2d(stg + p * kPatch, &tmX, col, row0_of(tile) + (ew & 3) * 32, &bars->x_full[h]);
                    }
                }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
        if (live) {
            // ------------------------------------------------------------ LayerNorm, SiLU, drain
            const int ew = warp - 4, quad = warp & 3, ch = ew >> 2;
            const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
            const int rr = quad * 32 + lane;          // this thread's row of the CTA's 128
            uint8_t *patches = stg + ew * (2 * kPatch);
            bool ok = true;
            auto wait = [&](uint64_t *bar, uint32_t parity) {
                ok = __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, err));
                return ok;
            };
            // one arrival per warp, when every lane's part is done
            auto arrive_leader = [&](uint64_t *bar) {
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive_cluster(tc::cluster_addr(bar, 0));
            };
            uint64_t xp[4][16];                       // x of the half row in groups of 32 columns, two columns each
            auto take_x = [&](auto half) {            // half H of tile n's x out of the staging area
                constexpr int H = decltype(half)::value;
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(patch_chunk(patches + p * kPatch, lane, j));
                        xp[2 * H + p][2 * j] = v.x; xp[2 * H + p][2 * j + 1] = v.y;
                    }
            };
            auto staging_free = [&] {
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&bars->stg_free);
            };
            {
                // (x has room for whole tiles of 128 rows; a tile's second 128 may lie wholly past them)
                const int64_t row = (int64_t)row0_of(tile0) + rr;
                const float *p = x + row * kD + ch * 128 + 64;
                if (row0_of(tile0) < M) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) load_x8(p + 8 * i, &xp[2 + i / 4][4 * (i % 4)]);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) xp[2 + i / 16][i % 16] = 0;
                }
            }
            if (wait(&bars->x_full[0], 0)) { take_x(Int<0>()); staging_free(); }
            // A quarter of the warp's part of a finished tile: x = O + b2, a patch of 32 rows x 32 columns handed to the TMA unit
            auto drain = [&](int tile, int gi, uint8_t *patch, bool reused) {
                const int cc = ch * 128 + gi * 32, row0 = row0_of(tile) + quad * 32;
                uint32_t r[32];
                tc::tmem_ld32(lane_addr + kColO + cc, r);
                tc::tmem_ld_wait();
                if (reused) {
                    if (lane == 0) tc::bulk_wait_read<1>();
                    __syncwarp();
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(b2s + cc + 4 * j);
                    *reinterpret_cast<ulonglong2 *>(patch_chunk(patch, lane, j)) =
                        make_ulonglong2(tc::add2(tc::pack2(r[4 * j], r[4 * j + 1]), q.x), tc::add2(tc::pack2(r[4 * j + 2], r[4 * j + 3]), q.y));
                }
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    if (row0 < M) tc::tma_store_2d(&tmX, patch, cc, row0);
                    tc::bulk_commit();
                }
            };
            int gc = 0, n = 0;
            // (a wait that ran out ends the loop at row_stats, for both warps of a quadrant: until there nothing more is waited for or stored)
            for (int tile = tile0; tile < n_tiles; tile += tile_step, ++n) {
                const bool more = tile + tile_step < n_tiles;
                // The tile before is drained column group by column group, and mid = x + att Wo^T + bo takes the place of what was
                // drained: the stores of one group are read while the next group's mid is computed.
                if (ok && n > 0) wait(&bars->o_full, (n - 1) & 1);
                RowStats st;
                if (ok) {
                    tc::tc_fence_after();
#pragma unroll
                    for (int gi = 0; gi < 4; ++gi) {
                        if (n > 0) drain(tile - tile_step, gi, patches + (gi & 1) * kPatch, gi > 1);
                        if (gi == 0) {
                            if (!wait(&bars->o1_full, n & 1)) break;
                            tc::tc_fence_after();
                        }
                        const int cc = ch * 128 + gi * 32;
                        uint32_t r[32];
                        tc::tmem_ld32(lane_addr + kColS + cc, r);
                        tc::tmem_ld_wait();
                        mid_group(r, xp[gi], bos + cc, gi, st);
                        tc::tmem_st32(lane_addr + kColO + cc, r);
                    }
                }
                float mean, rstd;
                ok = row_stats(st, stat, quad, ch, rr, eps, mean, rstd, ok);
                if (!ok) break;
                tc::tmem_st_wait();
                normalise(lane_addr + kColO + ch * 128, gs, bs, mean, rstd, sA, ch, rr);
                tc::fence_proxy_async();              // generic-proxy writes of the tile before the tensor core reads it
                arrive_leader(&bars->a_ready);
                if (n > 0 && lane == 0) {
                    tc::bulk_wait_read<0>();          // the drain's patches have been read
                    tc::mbar_arrive(&bars->stg_free);
                }

                for (int c = 0; c < nc; ++c) {
                    const int hb = (gc + c) & 1;
                    if (!wait(&bars->s_full[hb], ((gc + c) >> 1) & 1)) break;
                    tc::tc_fence_after();
                    silu_chunk(lane_addr + kColS + hb * kChunk + ch * 64, b1s + c * kChunk + ch * 64);
                    tc::tmem_st_wait();
                    arrive_leader(&bars->h_full[hb]);
                    // the next tile's x, while the tensor pipe works on what is queued
                    if (more && c == (nc - 1) / 2) {
                        if (!wait(&bars->x_full[0], (n + 1) & 1)) break;
                        take_x(Int<0>());
                        staging_free();
                    }
                    if (more && c == nc - 1) {
                        if (!wait(&bars->x_full[1], n & 1)) break;
                        take_x(Int<1>());
                    }
                }
                gc += nc;
            }
            if (ok && n > 0 && wait(&bars->o_full, (n - 1) & 1)) {          // the last tile
                tc::tc_fence_after();
#pragma unroll 1
                for (int gi = 0; gi < 4; ++gi)        // (the weight ring is idle: no patch has to wait for its last store)
                    drain(tile0 + (n - 1) * tile_step, gi, gi < 2 ? patches + gi * kPatch : sW + (2 * ew + gi - 2) * kPatch, false);
            }
            if (lane == 0) tc::bulk_wait_read<0>();   // the grid's completion covers the writes
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();                               // the peer no longer signals this CTA's barriers or uses its operands
    if (warp == 1) tc::tmem_dealloc_pair(tmem_base, kTmemCols);
}

}  // namespace

cudaError_t launch_ffn_pair(const FfnMaps &w, const CUtensorMap &tmX, const float *x, const float *g, const float *b, const float *b1, const float *b2,
                            const CUtensorMap &tmAtt, const float *bo, int64_t M, int d_ff, float eps, int *err, cudaStream_t stream)
{
    static PerDeviceValue pairs_of;                   // pairs that can be resident at once
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int pairs = pairs_of.get(dev);
    if (pairs == 0) {
        e = cudaFuncSetAttribute(ffn_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        cudaFuncAttributes attrs{};
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&attrs, ffn_pair_kernel);
        if (e == cudaSuccess && attrs.numRegs * kThreads < kOtherRegs * (kThreads - kEpiThreads) + kEpiRegs * kEpiThreads) e = cudaErrorInvalidValue;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(64); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kSmemBytes;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&pairs, ffn_pair_kernel, &cfg);
        if (e != cudaSuccess) return e;
        if (pairs < 1) return cudaErrorLaunchOutOfResources;
        pairs_of.set(dev, pairs);
    }
    const int64_t tiles = (M + 2 * kRows - 1) / (2 * kRows);
    const unsigned workers = (unsigned)(tiles < pairs ? tiles : pairs);
    return launch_dependent(ffn_pair_kernel, dim3(2 * workers), dim3(kThreads), (size_t)kSmemBytes, stream, 2, w.w1_half, w.w2, tmX, tmAtt, w.wo, x, g, b, b1,
                            b2, bo, M, d_ff, eps, err);
}

}  // namespace relaygr
