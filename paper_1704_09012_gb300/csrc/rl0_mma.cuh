// rl0_mma.cuh -- the learned column scorer's network (16 -> 32 -> 32 -> 1, ReLU)
// on the tensor cores: warp-level mma.sync m16n8k16 with BF16 operands and FP32
// accumulation, 16 rows (candidates or training samples) per warp.  Not part of
// the ABI.
//
// Precision.  An FP32 value x is split into three BF16 parts, x1 = bf16(x),
// x2 = bf16(x - x1), x3 = bf16(x - x1 - x2), which together carry its 24-bit
// significand; x1 + x2 + x3 = x unless x is below the BF16 normal range.  A
// product of such a part with a BF16 weight is exact in FP32, so a layer
// computed as sum_parts (x_p . W) differs from the FP32 dot product only by
// the FP32 accumulation's rounding.  The decoder's weights are BF16 already;
// FP32 master weights (training) are split the same way and the six products
// of parts whose ranks add up to at most 4 are kept (the rest are below 2^-24
// relative).
//
// Fragment layouts of mma.sync.m16n8k16 (PTX ISA): with g = lane / 4 and
// q = lane % 4, A (16 x 16, row-major) holds rows g and g + 8, columns 2q, 2q+1,
// 2q+8, 2q+9; B (16 x 8) holds rows (k) 2q, 2q+1, 2q+8, 2q+9 of column (n) g;
// C/D (16 x 8) holds rows g and g + 8, columns 2q and 2q+1.  So layer 1's
// accumulators over hidden units 16kk .. 16kk+15 (two n-tiles) are, entry for
// entry, layer 2's A fragment for k-step kk: no data moves between layers.
#pragma once

#include <cuda_bf16.h>

#include "rl0_device.cuh"

__device__ __forceinline__ unsigned bf16x2_bits(__nv_bfloat16 lo, __nv_bfloat16 hi)
{
    return (unsigned)__bfloat16_as_ushort(lo) | ((unsigned)__bfloat16_as_ushort(hi) << 16);
}

// x = p[0] + p[1] + p[2] in BF16 parts (round to nearest at each step)
__device__ __forceinline__ void split3(float x, __nv_bfloat16 *p)
{
    p[0] = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(p[0]);
    p[1] = __float2bfloat16_rn(r1);
    p[2] = __float2bfloat16_rn(r1 - __bfloat162float(p[1]));
}

// d += a . b, m16n8k16, BF16 x BF16 -> FP32
__device__ __forceinline__ void mma_bf16_16816(float *d, const unsigned *a, const unsigned *b)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// A fragments (three parts) of a 16 x 16 FP32 tile given its values at this
// lane's positions: v[0..1] row g cols 2q..2q+1, v[2..3] row g+8 same cols,
// v[4..5] row g cols 2q+8..2q+9, v[6..7] row g+8 same cols.
__device__ __forceinline__ void a_frag_split3(const float *v, unsigned a[3][4])
{
    __nv_bfloat16 p[8][3];
#pragma unroll
    for (int e = 0; e < 8; ++e) split3(v[e], p[e]);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        a[s][0] = bf16x2_bits(p[0][s], p[1][s]);
        a[s][1] = bf16x2_bits(p[2][s], p[3][s]);
        a[s][2] = bf16x2_bits(p[4][s], p[5][s]);
        a[s][3] = bf16x2_bits(p[6][s], p[7][s]);
    }
}

// B fragment of the BF16 matrix W (row-major, ldw columns; rows k0 .., columns n0 ..)
__device__ __forceinline__ void b_frag_bf16(const __nv_bfloat16 *W, int ldw, int k0, int n0, unsigned b[2])
{
    const int g = (threadIdx.x & 31) >> 2, q = threadIdx.x & 3;
    b[0] = bf16x2_bits(W[(k0 + 2 * q) * ldw + n0 + g], W[(k0 + 2 * q + 1) * ldw + n0 + g]);
    b[1] = bf16x2_bits(W[(k0 + 2 * q + 8) * ldw + n0 + g], W[(k0 + 2 * q + 9) * ldw + n0 + g]);
}

// d += a . b for two FP32 operands in three BF16 parts each: the six part
// products whose ranks add up to at most 4, smallest first.
__device__ __forceinline__ void mma_split3x3(float *d, const unsigned a[3][4], const unsigned b[3][2])
{
    mma_bf16_16816(d, a[2], b[0]);
    mma_bf16_16816(d, a[1], b[1]);
    mma_bf16_16816(d, a[0], b[2]);
    mma_bf16_16816(d, a[1], b[0]);
    mma_bf16_16816(d, a[0], b[1]);
    mma_bf16_16816(d, a[0], b[0]);
}

// The network's BF16 parameters where a warp reads them: in global memory in
// the order of rl0.h (W1 16x32 input-major, b1, W2 32x32, b2, w3, b3), ...
struct MlpGlobal {
    const __nv_bfloat16 *wb;
    // B fragment of n-tile nt of layer 1 (i = nt), of k-step kk and n-tile nt of layer 2 (i = 4 + 4 kk + nt)
    __device__ __forceinline__ void frag(int i, unsigned b[2]) const
    {
        if (i < 4) b_frag_bf16(wb + RL0_OFF_W1, RL0_HID, 0, 8 * i, b);
        else b_frag_bf16(wb + RL0_OFF_W2, RL0_HID, 16 * ((i - 4) >> 2), 8 * ((i - 4) & 3), b);
    }
    __device__ __forceinline__ float2 pair(int off, int u) const   // units u, u + 1 of the vector at off
    {
        return make_float2(__bfloat162float(wb[off + u]), __bfloat162float(wb[off + u + 1]));
    }
    __device__ __forceinline__ float b3() const { return __bfloat162float(wb[RL0_OFF_B3]); }
};

// ... or packed once per CTA in shared memory: every lane's fragment in one
// 8-byte word, the vectors in FP32.  From global memory a tile of 16 rows takes
// 48 two-byte loads of four cache lines each for the fragments and 25 more.
// Packed, and with the features' seven smallest deviations kept in registers
// (rl0_device.cuh): learned decodes at n = 60000, d = 8 1331 -> 1159 us, at n = 201716,
// d = 9 1047 -> 906 us, at n = 2^22, d = 7 (gathers from L2) 33.5 -> 32.6 ms; with few
// candidates (n = 15306) no change, 442 and 446 us.
struct MlpPacked {
    uint2 w[12][32];
    float2 b1[RL0_HID / 2], b2[RL0_HID / 2], w3[RL0_HID / 2];
    float b3v;
    __device__ __forceinline__ void frag(int i, unsigned b[2]) const
    {
        const uint2 v = w[i][threadIdx.x & 31];
        b[0] = v.x;
        b[1] = v.y;
    }
    __device__ __forceinline__ float2 pair(int off, int u) const
    {
        const float2 *p = off == RL0_OFF_B1 ? b1 : off == RL0_OFF_B2 ? b2 : w3;
        return p[u >> 1];
    }
    __device__ __forceinline__ float b3() const { return b3v; }
};

// Fills P (shared) with nt threads, a multiple of 32; a barrier follows before it is read.
__device__ __forceinline__ void mlp_pack(MlpPacked &P, const __nv_bfloat16 *wb, int tid, int nt)
{
    const MlpGlobal G{wb};
    for (int i = tid >> 5; i < 12; i += nt >> 5) {
        unsigned b[2];
        G.frag(i, b);
        P.w[i][tid & 31] = make_uint2(b[0], b[1]);
    }
    if (tid < RL0_HID / 2) {
        P.b1[tid] = G.pair(RL0_OFF_B1, 2 * tid);
        P.b2[tid] = G.pair(RL0_OFF_B2, 2 * tid);
        P.w3[tid] = G.pair(RL0_OFF_W3, 2 * tid);
    }
    if (tid == 0) P.b3v = G.b3();
}

// The same in two halves for a CTA of at least 384 threads: the loads (a thread's
// fragment and vector words, in registers), and the stores into P.
struct MlpSlice {
    unsigned b[2];
    float2 v;
    float b3v;
};

__device__ __forceinline__ void mlp_fetch(MlpSlice &L, const __nv_bfloat16 *wb, int tid)
{
    const MlpGlobal G{wb};
    const int lane = tid & 31, i = tid >> 5;
    if (i < 12) G.frag(i, L.b);
    // warps 0-2: b1, b2, w3
    if (i < 3 && lane < RL0_HID / 2) L.v = G.pair(i == 0 ? RL0_OFF_B1 : i == 1 ? RL0_OFF_B2 : RL0_OFF_W3, 2 * lane);
    if (tid == 0) L.b3v = G.b3();
}

__device__ __forceinline__ void mlp_store(MlpPacked &P, const MlpSlice &L, int tid)
{
    const int lane = tid & 31, i = tid >> 5;
    if (i < 12) P.w[i][lane] = make_uint2(L.b[0], L.b[1]);
    if (i < 3 && lane < RL0_HID / 2) (i == 0 ? P.b1 : i == 1 ? P.b2 : P.w3)[lane] = L.v;
    if (tid == 0) P.b3v = L.b3v;
}

// Logits of 16 rows with the parameters W (MlpGlobal or MlpPacked: the same
// arithmetic in the same order).  f(r, i) gives feature i of row r
// (rows 0..15 of this warp's tile).  Every lane of the warp calls it; lane
// 4g + q returns in *lo / *hi the logits of rows g and g + 8 (the same in the
// four lanes of a quad).
template <class FeatFn, class Params>
__device__ __forceinline__ void warp_mlp_logits16(FeatFn f, const Params &W, float *lo, float *hi)
{
    const int g = (threadIdx.x & 31) >> 2, q = threadIdx.x & 3;
    // layer 1: z1 = F W1 + b1 (K = 16, four n-tiles of 8 hidden units)
    unsigned a1[3][4];
    {
        float v[8];
        v[0] = f(g, 2 * q);
        v[1] = f(g, 2 * q + 1);
        v[2] = f(g + 8, 2 * q);
        v[3] = f(g + 8, 2 * q + 1);
        v[4] = f(g, 2 * q + 8);
        v[5] = f(g, 2 * q + 9);
        v[6] = f(g + 8, 2 * q + 8);
        v[7] = f(g + 8, 2 * q + 9);
        a_frag_split3(v, a1);
    }
    float c1[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const float2 b = W.pair(RL0_OFF_B1, 8 * nt + 2 * q);
        c1[nt][0] = b.x;
        c1[nt][1] = b.y;
        c1[nt][2] = b.x;
        c1[nt][3] = b.y;
        unsigned bw[2];
        W.frag(nt, bw);
#pragma unroll
        for (int s = 0; s < 3; ++s) mma_bf16_16816(c1[nt], a1[s], bw);
    }
    // layer 2: z2 = relu(z1) W2 + b2 (K = 32 in two k-steps)
    float c2[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const float2 b = W.pair(RL0_OFF_B2, 8 * nt + 2 * q);
        c2[nt][0] = b.x;
        c2[nt][1] = b.y;
        c2[nt][2] = b.x;
        c2[nt][3] = b.y;
    }
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[e] = fmaxf(c1[2 * kk][e], 0.0f);
            v[4 + e] = fmaxf(c1[2 * kk + 1][e], 0.0f);
        }
        unsigned a2[3][4];
        a_frag_split3(v, a2);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            unsigned bw[2];
            W.frag(4 + 4 * kk + nt, bw);
#pragma unroll
            for (int s = 0; s < 3; ++s) mma_bf16_16816(c2[nt], a2[s], bw);
        }
    }
    // layer 3: relu(z2) . w3 + b3, the quad's four column pairs added by shuffles
    float sl = 0.0f, sh = 0.0f;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const float2 w = W.pair(RL0_OFF_W3, 8 * nt + 2 * q);
        sl = fmaf(fmaxf(c2[nt][0], 0.0f), w.x, sl);
        sl = fmaf(fmaxf(c2[nt][1], 0.0f), w.y, sl);
        sh = fmaf(fmaxf(c2[nt][2], 0.0f), w.x, sh);
        sh = fmaf(fmaxf(c2[nt][3], 0.0f), w.y, sh);
    }
    sl += __shfl_xor_sync(0xffffffffu, sl, 1);
    sl += __shfl_xor_sync(0xffffffffu, sl, 2);
    sh += __shfl_xor_sync(0xffffffffu, sh, 1);
    sh += __shfl_xor_sync(0xffffffffu, sh, 2);
    const float b3 = W.b3();
    *lo = sl + b3;
    *hi = sh + b3;
}
