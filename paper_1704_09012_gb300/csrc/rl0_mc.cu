// rl0_mc.cu -- Monte-Carlo check of the posteriors p_z and p_e (arXiv
// 1704.09012, Section "Comparison with empirical probabilities", Fig. 3) with
// the library's own FP32 posterior series: binned counts of the events
// "y_i = 0" over the rows and "y_i = y_l" over the row pairs of each column,
// beside the sum of the posterior the decoder assigns to each sample.
//
// Integer histograms only, so the counts do not depend on scheduling.  A CTA
// keeps C copies of each bin's counters in shared memory, lane l of a warp using
// copy l mod C (a copy per lane for up to 192 bins: the lanes of a warp never
// meet, where most samples fall into few bins), as 32-bit words: the samples, the
// events, and the posteriors' 2^-32 units in their low 16 bits and the rest.  They
// are added to the 64-bit bins in global memory before a word can overflow.
#include <algorithm>
#include <cmath>

#include "rl0_common.cuh"
#include "rl0_device.cuh"

#define RL0_MC_MAX_BINS 1024
#define RL0_MC_NT 256
#define RL0_MC_WORDS 4                   // counters per bin
#define RL0_MC_SMEM 98304                // shared memory per CTA: two fit an SM

namespace {

struct McHist {
    unsigned *sh;                        // [(bin * RL0_MC_WORDS + word) * C + copy]
    int nbins, C, copy;
};

__device__ __forceinline__ void mc_add(const McHist &H, float a, bool event, float p)
{
    unsigned *h = H.sh + (unsigned)((int)a * RL0_MC_WORDS * H.C + H.copy);
    // p in [0, 1]; scaling by 2^32 is exact, the conversion rounds to nearest even
    const unsigned long long f = __float2ull_rn(p * 4294967296.0f);
    atomicAdd(h, 1u);
    if (event) atomicAdd(h + H.C, 1u);
    atomicAdd(h + 2 * H.C, (unsigned)f & 0xffffu);
    atomicAdd(h + 3 * H.C, (unsigned)(f >> 16));
}

// The CTA's counters to global memory, and to zero.  Every thread calls it.
__device__ __forceinline__ void mc_flush(const McHist &H, unsigned long long *out)
{
    __syncthreads();
    for (int b = threadIdx.x; b < H.nbins; b += blockDim.x) {
        unsigned long long v[RL0_MC_WORDS];
#pragma unroll
        for (int w = 0; w < RL0_MC_WORDS; ++w) {
            v[w] = 0ull;
            unsigned *h = H.sh + (unsigned)((b * RL0_MC_WORDS + w) * H.C);
            for (int c = 0; c < H.C; ++c) {
                const int q = (c + b) & (H.C - 1);       // (C is a power of two: spread over the banks)
                v[w] += h[q];
                h[q] = 0u;
            }
        }
        if (v[0]) {
            atomicAdd(&out[3 * b], v[0]);
            if (v[1]) atomicAdd(&out[3 * b + 1], v[1]);
            atomicAdd(&out[3 * b + 2], v[2] + (v[3] << 16));
        }
    }
    __syncthreads();
}

// Steps between flushes: a step adds at most RL0_MC_NT / C times `each` samples to
// one copy of a bin, each at most 2^16 to a word, and a word stays below 2^32.
__device__ __forceinline__ int mc_steps(int C, int each) { return max(1, (65536 / RL0_MC_NT * C - 1) / each); }

__device__ __forceinline__ McHist mc_open(unsigned *sh, int nbins, int C)
{
    for (int e = threadIdx.x; e < nbins * RL0_MC_WORDS * C; e += blockDim.x) sh[e] = 0u;
    __syncthreads();
    return McHist{sh, nbins, C, (int)(threadIdx.x & (C - 1))};
}

// Rows: bin |yhat_i|; event y0_i == 0; posterior p_breve_z(yhat_i).
__global__ void __launch_bounds__(RL0_MC_NT) k_mc_rows(int m, const float *__restrict__ y0,
                                                       const float *__restrict__ yh, Series pz, int nbins, int C,
                                                       float inv_w, unsigned long long *hz)
{
    extern __shared__ unsigned sh[];
    const McHist H = mc_open(sh, nbins, C);
    const int every = mc_steps(C, 1);
    int steps = 0;
    for (unsigned i0 = blockIdx.x * RL0_MC_NT; i0 < (unsigned)m; i0 += gridDim.x * RL0_MC_NT) {   // (may pass 2^31)
        const unsigned i = i0 + threadIdx.x;
        if (i < (unsigned)m) {
            const float w = yh[i], z = y0[i];
            const float a = fabsf(w) * inv_w;
            if (a < (float)nbins) mc_add(H, a, z == 0.0f, series_eval(pz, w));
        }
        if (++steps >= every) {
            mc_flush(H, hz);
            steps = 0;
        }
    }
    mc_flush(H, hz);
}

// Row pairs of every column (rows ascending, s < l): bin |yhat_s - yhat_l|;
// event y0_s == y0_l; posterior p_breve_e(yhat_s - yhat_l).  One thread per
// column, its d values in registers (slot-major row ids: coalesced).  n = 2^20,
// d = 7 (22 M pairs), 64 bins: the call took 444 us with three 64-bit atomics per
// pair on one copy of the bins, now 206, 187 of them here (issue: half the slots are
// busy, the warps wait for instructions of the unrolled pairs and for the queue of
// shared-memory operations).  Two gathers per row: with (yhat, y0)
// written side by side by the row kernel, one gather, it took 183, but the pairs
// need memory of the call's own for that.  The expander's workspace is not it (a
// decode, or another of these calls, may run on another stream), and a
// stream-ordered allocation takes 200 us in every call that is waited for.
template <int DMAX>
__global__ void __launch_bounds__(RL0_MC_NT) k_mc_pairs(int n, int d, const int32_t *__restrict__ rows_sm,
                                                        const float *__restrict__ y0, const float *__restrict__ yh,
                                                        Series pe, int nbins, int C, float inv_w,
                                                        unsigned long long *he)
{
    extern __shared__ unsigned sh[];
    const McHist H = mc_open(sh, nbins, C);
    const int every = mc_steps(C, max(1, d * (d - 1) / 2));
    int steps = 0;
    for (unsigned j0 = blockIdx.x * RL0_MC_NT; j0 < (unsigned)n; j0 += gridDim.x * RL0_MC_NT) {
        const unsigned j = j0 + threadIdx.x;
        if (j < (unsigned)n) {
            float2 v[DMAX];
#pragma unroll
            for (int s = 0; s < DMAX; ++s) {
                v[s] = make_float2(0.0f, 0.0f);
                if (s < d) {
                    const int i = __ldg(rows_sm + (size_t)s * n + j);
                    v[s] = make_float2(__ldg(yh + i), __ldg(y0 + i));
                }
            }
#pragma unroll
            for (int s = 0; s < DMAX; ++s) {
#pragma unroll
                for (int l = s + 1; l < DMAX; ++l) {
                    const float D = v[s].x - v[l].x;
                    const float a = fabsf(D) * inv_w;
                    if (l < d && a < (float)nbins) mc_add(H, a, v[s].y == v[l].y, series_eval(pe, D));
                }
            }
        }
        if (++steps >= every) {
            mc_flush(H, he);
            steps = 0;
        }
    }
    mc_flush(H, he);
}

}  // namespace

extern "C" int rl0_posterior_mc(const rl0_expander *A, const float *y0_dev, const float *yhat_dev, int64_t k,
                                double sigma_s, double sigma_n, int nbins, double wz_max, double we_max,
                                uint64_t *hz_dev, uint64_t *he_dev, void *cuda_stream)
{
    if (!A || !y0_dev || !yhat_dev || !hz_dev || !he_dev) return RL0_ERR_INVALID_ARG;
    if (k < 1 || k > A->m || !(sigma_s > 0.0) || !(sigma_n > 0.0) || nbins < 1 || nbins > RL0_MC_MAX_BINS ||
        !(wz_max > 0.0) || !(we_max > 0.0))
        return RL0_ERR_INVALID_ARG;
    int rc = rl0_set_device_of(A);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // the decoder's posterior series for this sparsity (Eqs. (pz_approx), (pe_approx), ell = 4)
    const double rho = (double)k / (double)A->m;
    const double s2 = sigma_s * sigma_s, n2 = sigma_n * sigma_n;
    const Series pz = rl0::to_device_series(rl0::make_series(A->d * rho, s2, n2, 4));
    const Series pe = rl0::to_device_series(rl0::make_series(2.0 * A->d * rho, s2, 2.0 * n2, 4));
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, A->device);
    nsm = std::max(nsm, 1);
    int C = 32;
    while (nbins * RL0_MC_WORDS * 4 * C > RL0_MC_SMEM) C /= 2;   // (C >= 4: nbins <= 1024)
    const int smem = nbins * RL0_MC_WORDS * 4 * C;
    const long long ctas = (long long)nsm * std::min(8, 2 * RL0_MC_SMEM / smem);
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if ((rc = rl0_cuda_err(cudaFuncSetAttribute(k_mc_rows, at, RL0_MC_SMEM)))) return rc;
    const int gr = (int)std::min<long long>(rl0_div_up(A->m, RL0_MC_NT), ctas);
    const int gp = (int)std::min<long long>(rl0_div_up(A->n, RL0_MC_NT), ctas);
    k_mc_rows<<<gr, RL0_MC_NT, smem, s>>>((int)A->m, y0_dev, yhat_dev, pz, nbins, C, (float)(nbins / wz_max),
                                          (unsigned long long *)hz_dev);
#define RL0_MP(D) do {                                                                                              \
        if ((rc = rl0_cuda_err(cudaFuncSetAttribute(k_mc_pairs<D>, at, RL0_MC_SMEM)))) return rc;                   \
        k_mc_pairs<D><<<gp, RL0_MC_NT, smem, s>>>((int)A->n, A->d, A->rows_sm, y0_dev, yhat_dev, pe, nbins, C,                  \
                                                  (float)(nbins / we_max), (unsigned long long *)he_dev);           \
    } while (0)
    if (A->d <= 8) RL0_MP(8);
    else if (A->d <= 16) RL0_MP(16);
    else RL0_MP(32);
#undef RL0_MP
    return rl0_cuda_err(cudaGetLastError());
}
