// What the forms of the fused out-proj + feed-forward kernel share: sizes and the query for resident clusters (all three: ffn_rows_tc.cu,
// ffn_tc.cu, ffn_pair_tc.cu), LayerNorm of whole rows in a warp (ffn_rows_tc.cu, embed_rows_tc.cu), and, for ffn_tc.cu and ffn_pair_tc.cu, the steps their eight
// epilogue warps take on one row (half) per thread.  Warp (quad, ch) owns TMEM lanes 32 quad .. + 31 and half ch of the columns.
// The row lives in TMEM and the steps walk it in rolled loops of 32 columns: a kernel of this kind runs a few microseconds per
// layer, between others that evict its instructions, so code that is executed once per tile costs its fetch from L2 (with
// everything unrolled over a row in registers, the first LayerNorm of a launch took 8000 clocks and later ones 3800).
#pragma once

#include "kernels.cuh"
#include "tc_common.cuh"

namespace relaygr {
namespace ffn {

constexpr int kD = 256;                              // d_model (O fills half of TMEM)
constexpr int kRows = 128, kChunk = 128, kMaxF = 2048;
constexpr int kEpiWarps = 8, kEpiThreads = 32 * kEpiWarps, kThreads = 128 + kEpiThreads;
constexpr int kABytes = kRows * kD * 2;              // 64 KB: four K blocks of [128 rows x 64] bf16, 128-byte swizzle
constexpr int kKBlock = kRows * 64 * 2;              // 16 KB
constexpr uint32_t kTmemCols = 512, kColO = 0, kColS = 256;      // S buffer i at kColS + 128 i; H in the first half of its S buffer's columns

// 16-byte chunk j of row r of a patch of 32 rows x 128 bytes in the 128-byte swizzle
__device__ __forceinline__ uint4 *patch_chunk(uint8_t *patch, int r, int j)
{
    return reinterpret_cast<uint4 *>(patch + r * 128 + ((j ^ (r & 7)) << 4));
}

// 32 bytes of x per lane, one whole sector each (a lane owns a row, so the rows of a warp are 1 KB apart)
__device__ __forceinline__ void load_x8(const float *p, uint64_t *v)
{
    asm volatile("ld.global.L1::no_allocate.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p) : "memory");
}

// Mean and sum of squared deviations of a row, built up 32 columns at a time (Chan, Golub, LeVeque: no cancellation, one pass).
struct RowStats { float mean = 0.f, m2 = 0.f; };

// 32 columns of a row: r = att Wo^T on entry, mid = x + att Wo^T + bo on return; gi = how many such groups came before.
__device__ __forceinline__ void mid_group(uint32_t (&r)[32], const uint64_t (&x)[16], const float *bo, int gi, RowStats &st)
{
    uint64_t v[16], s0 = 0, s1 = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(bo + 4 * j);
        v[2 * j] = tc::add2(tc::add2(x[2 * j], tc::pack2(r[4 * j], r[4 * j + 1])), q.x);
        v[2 * j + 1] = tc::add2(tc::add2(x[2 * j + 1], tc::pack2(r[4 * j + 2], r[4 * j + 3])), q.y);
        s0 = tc::add2(s0, v[2 * j]); s1 = tc::add2(s1, v[2 * j + 1]);
        tc::unpack2(v[2 * j], r[4 * j], r[4 * j + 1]);
        tc::unpack2(v[2 * j + 1], r[4 * j + 2], r[4 * j + 3]);
    }
    float a, b;
    tc::unpack2(tc::add2(s0, s1), a, b);
    const float gmean = (a + b) * (1.f / 32.f);
    const uint64_t nm = tc::pack2(-gmean, -gmean);
    s0 = s1 = 0;
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        const uint64_t d0 = tc::add2(v[j], nm), d1 = tc::add2(v[j + 1], nm);
        s0 = tc::fma2(d0, d0, s0); s1 = tc::fma2(d1, d1, s1);
    }
    tc::unpack2(tc::add2(s0, s1), a, b);
    const float delta = gmean - st.mean, w = 1.f / (float)(gi + 1);
    st.mean += delta * w;
    st.m2 += (a + b) + delta * delta * (32.f * (float)gi * w);
}

// The statistics of the whole row from its two halves (the two warps of a quadrant exchange them through `stat`): mean and 1 / std.
// ok: this warp's waits so far succeeded; returns whether both warps' did.
__device__ __forceinline__ bool row_stats(const RowStats &st, float2 *stat, int quad, int ch, int rr, float eps, float &mean, float &rstd, bool ok)
{
    stat[ch * kRows + rr] = make_float2(st.mean, st.m2);
    ok = tc::pair_all(1 + quad, ok);                  // the two warps that share these 32 rows
    const float2 o = stat[(ch ^ 1) * kRows + rr];
    mean = 0.5f * (st.mean + o.x);
    const float diff = st.mean - o.x;
    rstd = rsqrtf((st.m2 + o.y + diff * diff * (0.25f * kD)) * (1.f / kD) + eps);
    return ok;
}

// LN(mid) of this thread's half row, from O's columns, as bf16 into the K-major tile sA (rows of 128 bytes per K block).
__device__ __forceinline__ void normalise(uint32_t o_cols, const float *gs, const float *bs, float mean, float rstd, uint8_t *sA, int ch, int rr)
{
    const uint64_t nmean2 = tc::pack2(-mean, -mean), rstd2 = tc::pack2(rstd, rstd);
#pragma unroll 1
    for (int gi = 0; gi < 4; ++gi) {
        const int c0 = ch * 128 + gi * 32;
        uint32_t r[32];
        tc::tmem_ld32(o_cols + gi * 32, r);
        tc::tmem_ld_wait();
        uint8_t *row = sA + (c0 >> 6) * kKBlock + rr * 128;
#pragma unroll
        for (int i = 0; i < 4; ++i) {                 // eight columns = one 16-byte chunk
            uint32_t y[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const ulonglong2 ga = *reinterpret_cast<const ulonglong2 *>(gs + c0 + 8 * i + 4 * e), ba = *reinterpret_cast<const ulonglong2 *>(bs + c0 + 8 * i + 4 * e);
                const uint64_t v0 = tc::pack2(r[8 * i + 4 * e], r[8 * i + 4 * e + 1]), v1 = tc::pack2(r[8 * i + 4 * e + 2], r[8 * i + 4 * e + 3]);
                y[2 * e] = tc::pack_bf16(tc::fma2(tc::mul2(tc::add2(v0, nmean2), rstd2), ga.x, ba.x));
                y[2 * e + 1] = tc::pack_bf16(tc::fma2(tc::mul2(tc::add2(v1, nmean2), rstd2), ga.y, ba.y));
            }
            const int j = ((c0 & 63) >> 3) + i;
            *reinterpret_cast<uint4 *>(row + ((j ^ (rr & 7)) << 4)) = make_uint4(y[0], y[1], y[2], y[3]);
        }
    }
}

// H = SiLU(S + b1) of this warp's 64 columns of S: bf16 over the first 32 of them.  b1_half holds b1 / 2.
__device__ __forceinline__ void silu_chunk(uint32_t s_cols, const float *b1_half)
{
    const uint64_t half2 = tc::pack2(0.5f, 0.5f);
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {                     // H of columns 32 p .. goes where S of columns 16 p .. was: read by now
        uint32_t r[32], pk[16];
        tc::tmem_ld32(s_cols + 32 * p, r);
        tc::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(b1_half + 32 * p + 4 * e);
            pk[2 * e] = tc::pack_bf16(tc::silu2_of_half(tc::fma2(tc::pack2(r[4 * e], r[4 * e + 1]), half2, q.x)));
            pk[2 * e + 1] = tc::pack_bf16(tc::silu2_of_half(tc::fma2(tc::pack2(r[4 * e + 2], r[4 * e + 3]), half2, q.y)));
        }
        tc::tmem_st16(s_cols + 16 * p, pk);
    }
}

__device__ __forceinline__ float sum8(const float4 (&v)[2]) { return ((v[0].x + v[0].y) + (v[0].z + v[0].w)) + ((v[1].x + v[1].y) + (v[1].z + v[1].w)); }
// Mean and 1 / std of N rows, eight columns of each per lane.  Two passes; the rows' shuffles overlap.
template <int N>
__device__ __forceinline__ void rows_stats(const float4 (&v)[N][2], float eps, float (&mean)[N], float (&rstd)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) mean[i] = sum8(v[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) mean[i] += __shfl_xor_sync(0xffffffffu, mean[i], o);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        mean[i] *= 1.f / kD;
        float sq = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float dx = v[i][h].x - mean[i], dy = v[i][h].y - mean[i], dz = v[i][h].z - mean[i], dw = v[i][h].w - mean[i];
            sq += (dx * dx + dy * dy) + (dz * dz + dw * dw);
        }
        rstd[i] = sq;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) rstd[i] += __shfl_xor_sync(0xffffffffu, rstd[i], o);
#pragma unroll
    for (int i = 0; i < N; ++i) rstd[i] = rsqrtf(rstd[i] * (1.f / kD) + eps);
}
__device__ __forceinline__ float4 normalised(const float4 &v, float mean, float rstd, const float4 &g, const float4 &b)
{
    return make_float4((v.x - mean) * rstd * g.x + b.x, (v.y - mean) * rstd * g.y + b.y, (v.z - mean) * rstd * g.z + b.z, (v.w - mean) * rstd * g.w + b.w);
}

// How many clusters of `cs` CTAs of a kernel with `smem` bytes can be resident at once on the current device (`dev`); asked once.  None
// (a device or a part of one without that many SMs side by side) is an answer, not an error: the caller takes another form.
template <typename K>
cudaError_t resident_clusters(K kernel, int cs, size_t smem, PerDeviceValue &known, int dev, int *out)
{
    *out = known.get(dev);
    if (*out != 0) {
        *out = *out > 0 ? *out : 0;                   // (-1: none)
        return cudaSuccess;
    }
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cs * 16); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(out, kernel, &cfg);
    if (e != cudaSuccess) return e;
    known.set(dev, *out > 0 ? *out : -1);
    return cudaSuccess;
}

}  // namespace ffn
}  // namespace relaygr
