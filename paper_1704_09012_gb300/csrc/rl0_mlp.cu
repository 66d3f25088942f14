// rl0_mlp.cu -- the learned column scorer's network: a 16 -> 32 -> 32 -> 1 MLP
// with ReLU hidden layers and a logistic output, trained with binary
// cross-entropy on candidate features logged from analytic Robust-l0 decodes
// (labels: the candidate update x_j + w lands on the true x_j).  FP32 master
// weights train here; decodes use a BF16 copy with FP32 accumulation, on the
// tensor cores (rl0_mma.cuh).
//
// The gradient is deterministic: each CTA of the gradient kernel writes its own
// partial (its tiles of 16 samples in index order), and a second kernel adds the
// partials in a fixed order.
#include <algorithm>
#include <cmath>
#include <cstring>

#include <cuda_bf16.h>

#include "rl0_common.cuh"
#include "rl0_device.cuh"
#include "rl0_mma.cuh"
#include "rl0_round.cuh"

#define CK(call)                                          \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return rl0_cuda_err(e_);   \
    } while (0)

// He-normal initial weights (std sqrt(2 / fan_in)), zero biases.  Normal
// deviates by Box-Muller from a 64-bit mixing hash of (seed, index).
__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_mlp_init(unsigned long long seed, float *w)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= RL0_MLP_PARAMS) return;
    float fan = 0.0f;
    if (p < RL0_OFF_B1) fan = RL0_NFEAT;
    else if (p >= RL0_OFF_W2 && p < RL0_OFF_B2) fan = RL0_HID;
    else if (p >= RL0_OFF_W3 && p < RL0_OFF_B3) fan = RL0_HID;
    if (fan == 0.0f) { w[p] = 0.0f; return; }
    const unsigned long long h = mix64(seed * 0x100000001B3ull + (unsigned long long)p);
    const double u1 = ((double)(h >> 40) + 1.0) / 16777216.0;
    const double u2 = (double)((h >> 16) & 0xFFFFFFull) / 16777216.0;
    const double z = sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
    w[p] = (float)(z * sqrt(2.0 / fan));
}

// Loss and gradient of the mean binary cross-entropy
//   L = (1/N) sum_s softplus(o_s) - y_s o_s,   dL/do_s = (sigmoid(o_s) - y_s) / N,
// on the tensor cores, a block of RL0_MLP_BLOCK samples at a time.  Warp w takes
// samples 16w .. 16w+15 through the forward pass (z1 = F W1 + b1, z2 = relu(z1)
// W2 + b2) and the backward pass (D2 = relu'(z2) dL/do w3^T, D1 = relu'(z1)
// (D2 W2^T)) as m16n8k16 products, every activation in its accumulator fragment,
// which is the next product's A fragment.  movmatrix then transposes the
// fragments whose samples become the contraction index, and the CTA forms
// dW1 = F^T D1 and dW2 = H1^T D2 (K = the block's samples, in order) as 12 output
// tiles of 16 x 8 from fragments in shared memory, and the vector terms
// (biases, w3) with FP32 sums in sample order.  Both operands of every product
// are FP32 split into three BF16 parts, each value once; the weights' parts come
// as packed B fragments (k_mlp_pack, k_mlp_reduce_adam).
//
// What bounds it is latency: one block's chain of products, with one block per
// SM and 32 blocks in a minibatch of 4096.  Splitting operands inside the
// products' loops (the weights by every warp, X and D by every output tile), a
// 4096-row minibatch took 34-39 us here, now 8.9 us.
#define RL0_MLP_BLOCK 128
#define RL0_MLP_WARPS (RL0_MLP_BLOCK / 16)
// CTAs of a pass over more blocks than that: the GB300's 152 SMs (one CTA with the
// gradient's shared memory fits each, four without).  Constants, not the device's
// count: they set the order of the sums, which is the same on any device.
#define RL0_MLP_GRAD_CTAS 152
#define RL0_MLP_LOSS_CTAS 608
#define RL0_MLP_FWD_FRAGS 12                                // W1: 4 n-tiles; W2: 2 k-steps x 4 n-tiles
#define RL0_MLP_FRAGS 20                                    // and W2^T: 2 k-steps x 4 n-tiles
#define RL0_MLP_FRAG_WORDS (RL0_MLP_FRAGS * 3 * 64)         // two words per lane, three parts
#define RL0_MLP_PITCH 1664                                  // floats per CTA partial
#define RL0_MLP_LDH 36                                      // row pitch of D1, D2, H2

// Shared memory of k_mlp_block: the vectors and the weights' fragments (all that
// a pass without the gradient uses), then, per 16-sample
// step, the A fragments of F^T and H1^T and the B fragments of D1 and D2.
struct __align__(16) MlpShared {
    double loss[RL0_MLP_WARPS];
    float vec[3 * RL0_HID + 4];                             // b1, b2, w3, b3
    uint2 frag[RL0_MLP_FRAGS * 3 * 32];
    uint4 at[RL0_MLP_WARPS][3][3][32];                      // [step][F, H1 units 0-15, 16-31][part][lane]
    uint2 bt[RL0_MLP_WARPS][8][3][32];                      // [step][D1 n-tiles 0-3, D2 n-tiles 0-3][part][lane]
    float D1[RL0_MLP_BLOCK * RL0_MLP_LDH], D2[RL0_MLP_BLOCK * RL0_MLP_LDH], H2[RL0_MLP_BLOCK * RL0_MLP_LDH];
    float DO[RL0_MLP_BLOCK];
};
static_assert(offsetof(MlpShared, frag) % 16 == 0 && offsetof(MlpShared, at) % 16 == 0, "16-byte copies");

__device__ __forceinline__ unsigned transpose8x8(unsigned a)
{
    unsigned d;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}

// The A fragment (three parts) of X^T given X's A fragment.
__device__ __forceinline__ void transpose_frag(const unsigned a[3][4], unsigned t[3][4])
{
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        t[p][0] = transpose8x8(a[p][0]);
        t[p][1] = transpose8x8(a[p][2]);
        t[p][2] = transpose8x8(a[p][1]);
        t[p][3] = transpose8x8(a[p][3]);
    }
}

// The A fragment of X^T (three parts, from X's) to shared memory, and back.
__device__ __forceinline__ void store_transposed(uint4 (*dst)[32], const unsigned a[3][4], int lane)
{
    unsigned t[3][4];
    transpose_frag(a, t);
#pragma unroll
    for (int p = 0; p < 3; ++p) dst[p][lane] = make_uint4(t[p][0], t[p][1], t[p][2], t[p][3]);
}

__device__ __forceinline__ void load_a(const uint4 (*src)[32], int lane, unsigned a[3][4])
{
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const uint4 v = src[p][lane];
        a[p][0] = v.x;
        a[p][1] = v.y;
        a[p][2] = v.z;
        a[p][3] = v.w;
    }
}

// The B fragments (K = the 16 samples) of the two n-tiles of 8 units that the A
// fragment a (16 samples x 16 units) holds, to dst[0] and dst[1].
__device__ __forceinline__ void store_b_pair(uint2 (*dst)[3][32], const unsigned a[3][4], int lane)
{
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        dst[0][p][lane] = make_uint2(transpose8x8(a[p][0]), transpose8x8(a[p][1]));
        dst[1][p][lane] = make_uint2(transpose8x8(a[p][2]), transpose8x8(a[p][3]));
    }
}

__device__ __forceinline__ void load_b(const uint2 (*src)[32], int lane, unsigned b[3][2])
{
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const uint2 v = src[p][lane];
        b[p][0] = v.x;
        b[p][1] = v.y;
    }
}

// d += a . b with b a packed B fragment (part p of this lane at b[32 p])
__device__ __forceinline__ void mma_split3_packed(float *d, const unsigned a[3][4], const uint2 *b)
{
    unsigned w[3][2];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const uint2 v = b[32 * p];
        w[p][0] = v.x;
        w[p][1] = v.y;
    }
    mma_split3x3(d, a, w);
}

// The packed fragments' 16-bit entries of entry (k, n) of fragment f's 16 x 8 tile.
__device__ __forceinline__ void frag_store(unsigned short *frag, int f, int k, int n, const __nv_bfloat16 *part)
{
    const int reg = (k & 15) >> 3, q = (k & 7) >> 1, lane = 4 * n + q;
#pragma unroll
    for (int p = 0; p < 3; ++p)
        frag[(((f * 3 + p) * 32 + lane) * 2 + reg) * 2 + (k & 1)] = __bfloat16_as_ushort(part[p]);
}

// Parameter p's value v into the packed fragments.
__device__ __forceinline__ void pack_param(unsigned short *frag, int p, float v)
{
    __nv_bfloat16 part[3];
    if (p < RL0_OFF_B1) {
        const int k = p / RL0_HID, n = p % RL0_HID;
        split3(v, part);
        frag_store(frag, n >> 3, k, n & 7, part);
    } else if (p >= RL0_OFF_W2 && p < RL0_OFF_B2) {
        const int i = (p - RL0_OFF_W2) / RL0_HID, o = (p - RL0_OFF_W2) % RL0_HID;
        split3(v, part);
        frag_store(frag, 4 + (i >> 4) * 4 + (o >> 3), i & 15, o & 7, part);
        frag_store(frag, 12 + (o >> 4) * 4 + (i >> 3), o & 15, i & 7, part);     // W2^T
    }
}

__global__ void k_mlp_pack(const float *w, unsigned short *frag)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < RL0_MLP_PARAMS) pack_param(frag, p, w[p]);
}

// GRAD: part[CTA][p] = sum of dL/dw_p over the CTA's blocks (block b to CTA
// b mod gridDim, added in order); LOSS: loss_part[CTA] = the sum of its samples'
// losses in FP64.  vec: feat is 8-byte aligned.
template <bool GRAD, bool LOSS>
__global__ void __launch_bounds__(RL0_MLP_WARPS * 32) k_mlp_block(const float *__restrict__ w,
                                                                  const unsigned *__restrict__ frag,
                                                                  const float *__restrict__ feat,
                                                                  const float *__restrict__ label, long long N, int vec,
                                                                  float *__restrict__ part, double *loss_part)
{
    constexpr int NF = GRAD ? RL0_MLP_FRAGS : RL0_MLP_FWD_FRAGS;
    extern __shared__ __align__(16) unsigned char dsm[];
    MlpShared &M = *(MlpShared *)dsm;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int g = lane >> 2, q = lane & 3;
    const long long nblocks = (N + RL0_MLP_BLOCK - 1) / RL0_MLP_BLOCK;
    // features (A fragment positions) and labels of this warp's rows g and g + 8 of block b
    float fv[8], yl = 0.0f, yh = 0.0f;
    auto load_block = [&](long long b) {
        const long long sl = b * RL0_MLP_BLOCK + 16 * wid + g, sh = sl + 8;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long long s = h ? sh : sl;
            float2 v0 = make_float2(0.0f, 0.0f), v1 = v0;
            if (s < N) {
                const float *src = feat + s * RL0_NFEAT + 2 * q;
                if (vec) {
                    v0 = __ldg((const float2 *)src);
                    v1 = __ldg((const float2 *)(src + 8));
                } else {
                    v0 = make_float2(src[0], src[1]);
                    v1 = make_float2(src[8], src[9]);
                }
            }
            fv[2 * h] = v0.x;
            fv[2 * h + 1] = v0.y;
            fv[4 + 2 * h] = v1.x;
            fv[5 + 2 * h] = v1.y;
        }
        yl = (sl < N) ? __ldg(label + sl) : 0.0f;
        yh = (sh < N) ? __ldg(label + sh) : 0.0f;
    };
    load_block(blockIdx.x);                                 // (training data: no kernel writes it)
    pdl_wait();                                             // the previous step's weights
    pdl_launch_dependents();
    for (int e = t; e < NF * 3 * 16; e += blockDim.x) ((uint4 *)M.frag)[e] = __ldcg((const uint4 *)frag + e);
    for (int e = t; e < 3 * RL0_HID + 1; e += blockDim.x)
        M.vec[e] = __ldcg(w + (e < RL0_HID ? RL0_OFF_B1 + e : (e < 2 * RL0_HID ? RL0_OFF_B2 + e - RL0_HID
                                                                               : RL0_OFF_W3 + e - 2 * RL0_HID)));
    __syncthreads();
    const uint2 *B = M.frag + lane;
    float *P = part + (size_t)blockIdx.x * RL0_MLP_PITCH;
    double lsum = 0.0, lp = 0.0;                            // loss: sum of max(o, 0) - y o, and prod(1 + e^-|o|) - 1
    int lcount = 0;
    for (long long b = blockIdx.x; b < nblocks; b += gridDim.x) {
        const long long sl = b * RL0_MLP_BLOCK + 16 * wid + g;
        const bool vl = sl < N, vh = sl + 8 < N;
        const float y0 = yl, y1 = yh;
        // ---- forward
        unsigned af[3][4];
        a_frag_split3(fv, af);
        if (b + gridDim.x < nblocks) load_block(b + gridDim.x);
        float c1[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const float b0 = M.vec[8 * nt + 2 * q], b1 = M.vec[8 * nt + 2 * q + 1];
            c1[nt][0] = b0;
            c1[nt][1] = b1;
            c1[nt][2] = b0;
            c1[nt][3] = b1;
            mma_split3_packed(c1[nt], af, B + 96 * nt);
        }
        float c2[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const float b0 = M.vec[RL0_HID + 8 * nt + 2 * q], b1 = M.vec[RL0_HID + 8 * nt + 2 * q + 1];
            c2[nt][0] = b0;
            c2[nt][1] = b1;
            c2[nt][2] = b0;
            c2[nt][3] = b1;
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                v[e] = fmaxf(c1[2 * kk][e], 0.0f);
                v[4 + e] = fmaxf(c1[2 * kk + 1][e], 0.0f);
            }
            unsigned ah[3][4];                              // relu(z1), units 16 kk .. 16 kk + 15
            a_frag_split3(v, ah);
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) mma_split3_packed(c2[nt], ah, B + 96 * (4 + 4 * kk + nt));
            if (GRAD) store_transposed(M.at[wid][1 + kk], ah, lane);
        }
        float ol = 0.0f, oh = 0.0f;                         // rows g and g + 8
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const float w0 = M.vec[2 * RL0_HID + 8 * nt + 2 * q], w1 = M.vec[2 * RL0_HID + 8 * nt + 2 * q + 1];
            ol = fmaf(fmaxf(c2[nt][0], 0.0f), w0, ol);
            ol = fmaf(fmaxf(c2[nt][1], 0.0f), w1, ol);
            oh = fmaf(fmaxf(c2[nt][2], 0.0f), w0, oh);
            oh = fmaf(fmaxf(c2[nt][3], 0.0f), w1, oh);
        }
        ol += __shfl_xor_sync(0xffffffffu, ol, 1);
        ol += __shfl_xor_sync(0xffffffffu, ol, 2);
        oh += __shfl_xor_sync(0xffffffffu, oh, 1);
        oh += __shfl_xor_sync(0xffffffffu, oh, 2);
        ol += M.vec[3 * RL0_HID];
        oh += M.vec[3 * RL0_HID];
        if (LOSS) {
            // softplus(o) = max(o, 0) + log(1 + e^-|o|); the logarithm of the product
            // of the factors is taken once per 256 of them (below 2^256)
            const bool mine = q == 0 ? vl : (q == 1 && vh);
            if (mine) {
                const double o = (double)(q == 0 ? ol : oh), y = (double)(q == 0 ? y0 : y1);
                const double e = exp(-fabs(o));
                lp = fma(e, 1.0 + lp, lp);
                lsum += (o > 0.0 ? o : 0.0) - y * o;
                if (++lcount == 256) {
                    lsum += log1p(lp);
                    lp = 0.0;
                    lcount = 0;
                }
            }
        }
        if (!GRAD) continue;
        const float dl = vl ? (1.0f / (1.0f + expf(-ol)) - y0) / (float)N : 0.0f;
        const float dh = vh ? (1.0f / (1.0f + expf(-oh)) - y1) / (float)N : 0.0f;
        const int r0 = 16 * wid;
        if (q == 0) {
            M.DO[r0 + g] = dl;
            M.DO[r0 + g + 8] = dh;
        }
        store_transposed(M.at[wid][0], af, lane);
        // ---- backward: D2 in c2's layout, D1 = relu'(z1) (D2 W2^T)
        float d1[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) d1[nt][e] = 0.0f;
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {                    // K = the 32 units of z2
            float v[8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int nt = 2 * kk + h;
                const float w0 = M.vec[2 * RL0_HID + 8 * nt + 2 * q], w1 = M.vec[2 * RL0_HID + 8 * nt + 2 * q + 1];
                v[4 * h] = (c2[nt][0] > 0.0f) ? dl * w0 : 0.0f;
                v[4 * h + 1] = (c2[nt][1] > 0.0f) ? dl * w1 : 0.0f;
                v[4 * h + 2] = (c2[nt][2] > 0.0f) ? dh * w0 : 0.0f;
                v[4 * h + 3] = (c2[nt][3] > 0.0f) ? dh * w1 : 0.0f;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int o = (r0 + g + ((e & 2) ? 8 : 0)) * RL0_MLP_LDH + 8 * nt + 2 * q + (e & 1);
                    M.D2[o] = v[4 * h + e];
                    M.H2[o] = fmaxf(c2[nt][e], 0.0f);
                }
            }
            unsigned ad[3][4];
            a_frag_split3(v, ad);
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) mma_split3_packed(d1[nt], ad, B + 96 * (12 + 4 * kk + nt));
            store_b_pair(M.bt[wid] + 4 + 2 * kk, ad, lane);
        }
#pragma unroll
        for (int mm = 0; mm < 2; ++mm) {
            float v[8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int nt = 2 * mm + h;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[4 * h + e] = (c1[nt][e] > 0.0f) ? d1[nt][e] : 0.0f;
                    M.D1[(r0 + g + ((e & 2) ? 8 : 0)) * RL0_MLP_LDH + 8 * nt + 2 * q + (e & 1)] = v[4 * h + e];
                }
            }
            unsigned a1[3][4];
            a_frag_split3(v, a1);
            store_b_pair(M.bt[wid] + 2 * mm, a1, lane);
        }
        __syncthreads();
        const bool add = b != blockIdx.x;                   // a later block of this CTA
        // ---- weight matrices: 4 tiles of dW1 (16 x 32) and 8 of dW2 (32 x 32), K = the
        // block's samples; warps 0-3 take two of them side by side, warps 4-7 one and a vector
        {
            const bool two = wid < 4;
            float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, acc2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            const int ta = wid, tb = two ? 8 + wid : wid;   // tiles 0-3: dW1; 4-7, 8-11: dW2 units 0-15, 16-31
#pragma unroll
            for (int ks = 0; ks < RL0_MLP_WARPS; ++ks) {
                unsigned a[3][4], bb[3][2];
                load_a(M.at[ks][ta >> 2], lane, a);
                load_b(M.bt[ks][ta < 4 ? ta : 4 + (ta & 3)], lane, bb);
                mma_split3x3(acc, a, bb);
                if (two) {
                    load_a(M.at[ks][2], lane, a);
                    load_b(M.bt[ks][4 + (tb & 3)], lane, bb);
                    mma_split3x3(acc2, a, bb);
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int row = g + ((e & 2) ? 8 : 0), c = 2 * q + (e & 1);
                const int pa = (ta < 4 ? RL0_OFF_W1 : RL0_OFF_W2) + row * RL0_HID + 8 * (ta & 3) + c;
                P[pa] = add ? P[pa] + acc[e] : acc[e];
                if (two) {
                    const int pb = RL0_OFF_W2 + (16 + row) * RL0_HID + 8 * (tb & 3) + c;
                    P[pb] = add ? P[pb] + acc2[e] : acc2[e];
                }
            }
        }
        // ---- vectors: db1, db2, dw3 (sums over samples in index order) and db3
        if (wid >= 4 && (wid < 7 || lane == 0)) {
            float acc = 0.0f;
            int po;
            if (wid == 4) {
                for (int s2 = 0; s2 < RL0_MLP_BLOCK; ++s2) acc += M.D1[s2 * RL0_MLP_LDH + lane];
                po = RL0_OFF_B1 + lane;
            } else if (wid == 5) {
                for (int s2 = 0; s2 < RL0_MLP_BLOCK; ++s2) acc += M.D2[s2 * RL0_MLP_LDH + lane];
                po = RL0_OFF_B2 + lane;
            } else if (wid == 6) {
                for (int s2 = 0; s2 < RL0_MLP_BLOCK; ++s2) acc = fmaf(M.H2[s2 * RL0_MLP_LDH + lane], M.DO[s2], acc);
                po = RL0_OFF_W3 + lane;
            } else {
                for (int s2 = 0; s2 < RL0_MLP_BLOCK; ++s2) acc += M.DO[s2];
                po = RL0_OFF_B3;
            }
            P[po] = add ? P[po] + acc : acc;
        }
        if (b + gridDim.x < nblocks) __syncthreads();       // the fragments are overwritten by the next block
    }
    if (LOSS) {
        lsum += log1p(lp);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0) M.loss[wid] = lsum;
        __syncthreads();
        if (t == 0) {
            double l = 0.0;
            for (int v = 0; v < RL0_MLP_WARPS; ++v) l += M.loss[v];
            loss_part[blockIdx.x] = l;
        }
    }
}

// Parameter p's gradient: the CTA partials added in CTA order, 16 loads in flight.
#define RL0_MLP_RED 32
__device__ __forceinline__ float sum_partials(const float *part, int nparts, int p)
{
    float acc = 0.0f;
    int b = 0;
    for (; b + 16 <= nparts; b += 16) {
        float x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) x[u] = __ldcg(part + (size_t)(b + u) * RL0_MLP_PITCH + p);
#pragma unroll
        for (int u = 0; u < 16; ++u) acc += x[u];
    }
    for (; b < nparts; ++b) acc += __ldcg(part + (size_t)b * RL0_MLP_PITCH + p);
    return acc;
}

// grad and the mean loss (NULL: none) from the CTA partials.
__global__ void __launch_bounds__(RL0_MLP_RED) k_mlp_grad_reduce(const float *part, int nparts, float *grad,
                                                                 const double *loss_part, double *loss, long long N)
{
    pdl_wait();
    const int p = blockIdx.x * RL0_MLP_RED + threadIdx.x;
    if (grad && p < RL0_MLP_PARAMS) grad[p] = sum_partials(part, nparts, p);
    if (loss && blockIdx.x == 0) {
        double l = 0.0;
        for (int b = threadIdx.x; b < nparts; b += 32) l += __ldcg(loss_part + b);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (threadIdx.x == 0) *loss = l / (double)N;
    }
}

// Adam (Kingma and Ba, 2015) with bias correction on the gradient the CTA
// partials add up to; the new weights go into the packed fragments as well.
// One thread per parameter, its partials 16 loads at a time; the launches overlap
// (features and moments load while the previous kernel finishes).  A 4096-row
// step, both kernels alone (ncu): 37 + 4.8 -> 8.9 + 4.3 us; two epochs over
// 400 003 rows with the final loss 8.33 -> 2.19 ms.
__global__ void __launch_bounds__(RL0_MLP_RED) k_mlp_reduce_adam(const float *part, int nparts, float *w, float *m,
                                                                 float *v, unsigned short *frag, int step, float lr,
                                                                 float b1, float b2, float eps)
{
    const int p = blockIdx.x * RL0_MLP_RED + threadIdx.x;
    if (p >= RL0_MLP_PARAMS) return;
    // (last written two kernels ago)
    const float m0 = __ldcg(m + p), v0 = __ldcg(v + p), w0 = __ldcg(w + p);
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    pdl_wait();                                             // this step's partials
    pdl_launch_dependents();
    const float gp = sum_partials(part, nparts, p);
    const float mp = fmaf(1.0f - b1, gp, b1 * m0);
    const float vp = fmaf((1.0f - b2) * gp, gp, b2 * v0);
    m[p] = mp;
    v[p] = vp;
    const float mh = mp / c1;
    const float vh = vp / c2;
    const float wn = w0 - lr * mh / (sqrtf(vh) + eps);
    w[p] = wn;
    pack_param(frag, p, wn);
}

__global__ void k_mlp_export(const float *w, __nv_bfloat16 *wb)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < RL0_MLP_PARAMS) wb[p] = __float2bfloat16_rn(w[p]);
}

// Logits of N feature rows with the BF16 parameters: the decoder's arithmetic
// (warp_mlp_logits16 on the tensor cores), one warp per 16 rows.
__global__ void __launch_bounds__(256) k_mlp_forward(const __nv_bfloat16 *wb, const float *feat, long long N,
                                                      float *logit)
{
    const long long r0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / 32 * 16;
    if (r0 >= N) return;                           // whole warps leave together
    auto f = [&](int r, int i) { return (r0 + r < N) ? feat[(r0 + r) * RL0_NFEAT + i] : 0.0f; };
    float lo, hi;
    warp_mlp_logits16(f, MlpGlobal{wb}, &lo, &hi);
    const int g = (threadIdx.x & 31) >> 2;
    if ((threadIdx.x & 3) == 0) {
        if (r0 + g < N) logit[r0 + g] = lo;
        if (r0 + g + 8 < N) logit[r0 + g + 8] = hi;
    }
}

// ---------------------------------------------------------------------------
// Host
// ---------------------------------------------------------------------------
static const unsigned kRedGrid = (RL0_MLP_PARAMS + RL0_MLP_RED - 1) / RL0_MLP_RED;

static int mlp_blocks(long long N) { return (int)((N + RL0_MLP_BLOCK - 1) / RL0_MLP_BLOCK); }

// The limit on dynamic shared memory (an attribute of the kernels, set before use).
static int mlp_smem_limit()
{
    const int sm = (int)sizeof(MlpShared);
    CK(cudaFuncSetAttribute((const void *)k_mlp_block<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    CK(cudaFuncSetAttribute((const void *)k_mlp_block<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    CK(cudaFuncSetAttribute((const void *)k_mlp_block<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
    return RL0_OK;
}

static int aligned8(const float *p) { return ((size_t)p & 7u) == 0; }

extern "C" int rl0_mlp_init(uint64_t seed, float *w_dev, void *cuda_stream)
{
    if (!w_dev) return RL0_ERR_INVALID_ARG;
    k_mlp_init<<<(RL0_MLP_PARAMS + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(seed, w_dev);
    CK(cudaGetLastError());
    return RL0_OK;
}

extern "C" int rl0_mlp_grad(const float *w_dev, const float *feat_dev, const float *label_dev, int64_t N,
                            float *grad_dev, double *loss_host, void *cuda_stream)
{
    if (!w_dev || !feat_dev || !label_dev || !grad_dev || N < 1) return RL0_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int rc = mlp_smem_limit();
    if (rc) return rc;
    const int grid = std::min(mlp_blocks(N), RL0_MLP_GRAD_CTAS);
    // one block: CTA partials, packed fragments, loss partials, the loss
    const size_t o_frag = (size_t)grid * RL0_MLP_PITCH * sizeof(float);
    const size_t o_lp = o_frag + RL0_MLP_FRAG_WORDS * sizeof(unsigned), o_ld = o_lp + (size_t)grid * sizeof(double);
    unsigned char *buf = nullptr;
    CK(cudaMallocAsync(&buf, o_ld + sizeof(double), s));
    float *part = (float *)buf;
    unsigned *frag = (unsigned *)(buf + o_frag);
    double *lp = (double *)(buf + o_lp), *ld = (double *)(buf + o_ld);
    k_mlp_pack<<<(RL0_MLP_PARAMS + 255) / 256, 256, 0, s>>>(w_dev, (unsigned short *)frag);
    k_mlp_block<true, true><<<grid, RL0_MLP_WARPS * 32, sizeof(MlpShared), s>>>(w_dev, frag, feat_dev, label_dev,
                                                                                 (long long)N, aligned8(feat_dev), part,
                                                                                 lp);
    k_mlp_grad_reduce<<<kRedGrid, RL0_MLP_RED, 0, s>>>(part, grid, grad_dev, lp, ld, (long long)N);
    rc = rl0_cuda_err(cudaGetLastError());
    double l = 0.0;
    if (!rc) rc = rl0_cuda_err(cudaMemcpyAsync(&l, ld, sizeof(double), cudaMemcpyDeviceToHost, s));
    cudaFreeAsync(buf, s);
    if (!rc) rc = rl0_cuda_err(cudaStreamSynchronize(s));
    if (loss_host) *loss_host = l;
    return rc;
}

extern "C" int rl0_mlp_train(float *w_dev, const float *feat_dev, const float *label_dev, int64_t N, int epochs,
                             int batch, float lr, void *wbf16_dev, double *loss_host, void *cuda_stream)
{
    if (!w_dev || !feat_dev || !label_dev || N < 1 || epochs < 1 || batch < 1 || !(lr > 0.0f))
        return RL0_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int rc = mlp_smem_limit();
    if (rc) return rc;
    // a minibatch: one block per CTA; the final loss: resident CTAs (no gradient: the
    // weights' fragments are all the shared memory they use)
    const int gmax = mlp_blocks(std::min<int64_t>(N, batch)), gall = std::min(mlp_blocks(N), RL0_MLP_LOSS_CTAS);
    // one block: CTA partials, packed fragments, Adam's moments, loss partials, the loss
    const size_t o_frag = (size_t)gmax * RL0_MLP_PITCH * sizeof(float);
    const size_t o_m = o_frag + RL0_MLP_FRAG_WORDS * sizeof(unsigned), o_v = o_m + RL0_MLP_PITCH * sizeof(float);
    const size_t o_lp = o_v + RL0_MLP_PITCH * sizeof(float), o_ld = o_lp + (size_t)gall * sizeof(double);
    unsigned char *buf = nullptr;
    CK(cudaMallocAsync(&buf, o_ld + sizeof(double), s));
    float *part = (float *)buf, *m = (float *)(buf + o_m), *v = (float *)(buf + o_v);
    unsigned *frag = (unsigned *)(buf + o_frag);
    double *lp = (double *)(buf + o_lp), *ld = (double *)(buf + o_ld);
    const int vec = aligned8(feat_dev);
    rc = rl0_cuda_err(cudaMemsetAsync(m, 0, 2 * RL0_MLP_PITCH * sizeof(float), s));
    int step = 0;
    if (!rc) {
        k_mlp_pack<<<(RL0_MLP_PARAMS + 255) / 256, 256, 0, s>>>(w_dev, (unsigned short *)frag);
        rc = rl0_cuda_err(cudaGetLastError());
    }
    for (int ep = 0; ep < epochs && !rc; ++ep) {
        for (int64_t b0 = 0; b0 < N && !rc; b0 += batch) {
            const long long nb = (N - b0 < batch) ? (N - b0) : batch;
            const int grid = mlp_blocks(nb);
            launch_pdl(k_mlp_block<true, false>, grid, RL0_MLP_WARPS * 32, sizeof(MlpShared), s, (const float *)w_dev,
                       (const unsigned *)frag, feat_dev + b0 * RL0_NFEAT, label_dev + b0, nb, vec, part,
                       (double *)nullptr);
            ++step;
            launch_pdl(k_mlp_reduce_adam, kRedGrid, RL0_MLP_RED, 0, s, (const float *)part, grid, w_dev, m, v,
                       (unsigned short *)frag, step, lr, 0.9f, 0.999f, 1e-8f);
            rc = rl0_cuda_err(cudaGetLastError());
        }
    }
    if (!rc) {
        // loss of the final weights over the whole set
        launch_pdl(k_mlp_block<false, true>, gall, RL0_MLP_WARPS * 32, offsetof(MlpShared, at), s, (const float *)w_dev,
                   (const unsigned *)frag, feat_dev, label_dev, (long long)N, vec, (float *)nullptr, lp);
        launch_pdl(k_mlp_grad_reduce, 1u, RL0_MLP_RED, 0, s, (const float *)nullptr, gall, (float *)nullptr,
                   (const double *)lp, ld, (long long)N);
        double l = 0.0;
        rc = rl0_cuda_err(cudaGetLastError());
        if (!rc) rc = rl0_cuda_err(cudaMemcpyAsync(&l, ld, sizeof(double), cudaMemcpyDeviceToHost, s));
        if (!rc && wbf16_dev)
            k_mlp_export<<<(RL0_MLP_PARAMS + 255) / 256, 256, 0, s>>>(w_dev, (__nv_bfloat16 *)wbf16_dev);
        if (!rc) rc = rl0_cuda_err(cudaStreamSynchronize(s));
        if (loss_host) *loss_host = l;
    }
    cudaFreeAsync(buf, s);
    cudaStreamSynchronize(s);
    return rc;
}

extern "C" int rl0_mlp_export(const float *w_dev, void *wbf16_dev, void *cuda_stream)
{
    if (!w_dev || !wbf16_dev) return RL0_ERR_INVALID_ARG;
    k_mlp_export<<<(RL0_MLP_PARAMS + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(w_dev,
                                                                                     (__nv_bfloat16 *)wbf16_dev);
    CK(cudaGetLastError());
    return RL0_OK;
}

extern "C" int rl0_mlp_forward(const void *wbf16_dev, const float *feat_dev, int64_t N, float *logit_dev,
                               void *cuda_stream)
{
    if (!wbf16_dev || !feat_dev || !logit_dev || N < 0) return RL0_ERR_INVALID_ARG;
    if (N == 0) return RL0_OK;
    // 16 rows per warp, 8 warps per block
    k_mlp_forward<<<(unsigned)((N + 127) / 128), 256, 0, (cudaStream_t)cuda_stream>>>(
        (const __nv_bfloat16 *)wbf16_dev, feat_dev, N, logit_dev);
    CK(cudaGetLastError());
    return RL0_OK;
}

// ---------------------------------------------------------------------------
// Training data: the candidates met along an analytic decode, labelled
// ---------------------------------------------------------------------------

// sum |v_i| in FP64, one block, fixed order
__global__ void k_l1_f64(const float *v, int n, double *out)
{
    __shared__ double sh[1024];
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += fabs((double)v[i]);
    const double r = group_sum_f64(acc, sh, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) *out = r;
}

// label of candidate e: the update x_hat_j + w lands within tol of x_true_j != 0
__global__ void k_label(const int32_t *meta, const float *omega, const float *xhat, const float *xtrue, int c,
                        float tol, float *label)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= c) return;
    const int j = meta[4 * e];
    const float xt = xtrue[j];
    const float prop = xhat[j] + omega[e];
    label[e] = (fabsf(prop - xt) <= tol && xt != 0.0f) ? 1.0f : 0.0f;
}

extern "C" int rl0_scorer_log(const rl0_expander *A, const float *y_dev, int64_t k, const rl0_params *params,
                              const float *xtrue_dev, float tol_sigma, int max_rounds, float *feat_dev,
                              float *label_dev, int64_t cap, int64_t *count_out, int *rounds_out,
                              void *cuda_stream)
{
    if (!A || !y_dev || !params || !xtrue_dev || !count_out || cap < 0 || (cap > 0 && (!feat_dev || !label_dev)) ||
        !(tol_sigma > 0.0f) || max_rounds < 2 || max_rounds > RL0_MAX_ROUNDS)
        return RL0_ERR_INVALID_ARG;
    if (params->scorer != 0 || params->adaptive_k) return RL0_ERR_UNSUPPORTED;
    if (!(params->sigma_n > 0.0)) return RL0_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int64_t n = A->n, m = A->m;
    // candidates of one round: at most one per (column, anchor slot)
    const int64_t per_round = std::min<int64_t>(n * A->d, (int64_t)0x7fffffff);
    float *xh = nullptr, *rh = nullptr, *xp = nullptr, *rp = nullptr, *om = nullptr, *ftmp = nullptr;
    int32_t *meta = nullptr;
    double *dl1 = nullptr;
    int rc = RL0_OK;
    auto alloc = [&](void **p, size_t bytes) {
        if (!rc) rc = rl0_cuda_err(cudaMallocAsync(p, bytes, s));
    };
    alloc((void **)&xh, n * sizeof(float));
    alloc((void **)&xp, n * sizeof(float));
    alloc((void **)&rh, m * sizeof(float));
    alloc((void **)&rp, m * sizeof(float));
    alloc((void **)&meta, per_round * 4 * sizeof(int32_t));
    alloc((void **)&om, per_round * sizeof(float));
    alloc((void **)&ftmp, per_round * RL0_NFEAT * sizeof(float));
    alloc((void **)&dl1, sizeof(double));
    if (!rc) rc = rl0_cuda_err(cudaMemsetAsync(xh, 0, n * sizeof(float), s));
    if (!rc) rc = rl0_cuda_err(cudaMemcpyAsync(rh, y_dev, m * sizeof(float), cudaMemcpyDeviceToDevice, s));
    double l1h = 0.0;
    if (!rc) {
        k_l1_f64<<<1, 1024, 0, s>>>(y_dev, (int)m, dl1);
        rc = rl0_cuda_err(cudaMemcpyAsync(&l1h, dl1, sizeof(double), cudaMemcpyDeviceToHost, s));
        if (!rc) rc = rl0_cuda_err(cudaStreamSynchronize(s));
    }
    // the noise floor E||eta||_1 = m sigma_n sqrt(2 / pi): the decode's stop level
    const double stop = (double)m * params->sigma_n * sqrt(2.0 / M_PI);
    const float tol = (float)(tol_sigma * params->sigma_n);
    int64_t total = 0;
    int rounds = 0;
    for (int r = 1; r < max_rounds && !rc; ++r) {
        int c = 0;
        rc = rl0_candidate_features(A, y_dev, k, params, r, xh, rh, ftmp, meta, om, (int)per_round, &c, cuda_stream);
        if (rc) break;
        const int64_t take = std::min<int64_t>(c, cap - std::min(cap, total));
        if (take > 0) {
            rc = rl0_cuda_err(cudaMemcpyAsync(feat_dev + total * RL0_NFEAT, ftmp, take * RL0_NFEAT * sizeof(float),
                                              cudaMemcpyDeviceToDevice, s));
            if (rc) break;
            k_label<<<(unsigned)((take + 255) / 256), 256, 0, s>>>(meta, om, xh, xtrue_dev, (int)take, tol,
                                                                  label_dev + total);
            rc = rl0_cuda_err(cudaGetLastError());
            if (rc) break;
        }
        total += c;
        double l1 = 0.0;
        rc = rl0_round_step(A, y_dev, k, params, r, xh, rh, xp, rp, nullptr, &l1, cuda_stream);
        if (rc) break;
        ++rounds;
        if (l1 < l1h) {                            // accept: ||r||_1 < ||r_hat||_1
            std::swap(xh, xp);
            std::swap(rh, rp);
            l1h = l1;
        }
        if (l1h <= stop) break;
    }
    for (void *p : {(void *)xh, (void *)rh, (void *)xp, (void *)rp, (void *)om, (void *)ftmp, (void *)meta,
                    (void *)dl1})
        if (p) cudaFreeAsync(p, s);
    const int rs = rl0_cuda_err(cudaStreamSynchronize(s));
    if (!rc) rc = rs;
    *count_out = total;
    if (rounds_out) *rounds_out = rounds;
    return rc;
}

extern "C" int rl0_mlp_params(void) { return RL0_MLP_PARAMS; }
