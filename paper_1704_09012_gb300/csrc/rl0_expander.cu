// rl0_expander.cu -- the expander matrix A of Def. 1.1 and the generating model
// GM(n,m,k,d,mu,nu) (Def. "Generating model", Fig. 1) on the GPU: drawing A,
// validating caller rows, the slot-major and CSR(A^T) copies, and the sketch
// y_hat = A x + eta.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <new>

#include "rl0_common.cuh"

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32 multiplies
// with the key advanced by the golden-ratio Weyl constants between rounds.
// ---------------------------------------------------------------------------
struct PhiloxOut {
    uint32_t v[4];
};

__device__ __forceinline__ PhiloxOut philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                   uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
        const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
        const uint32_t o0 = hi1 ^ c1 ^ k0, o2 = hi0 ^ c3 ^ k1;
        c0 = o0; c1 = lo1; c2 = o2; c3 = lo0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    PhiloxOut r;
    r.v[0] = c0; r.v[1] = c1; r.v[2] = c2; r.v[3] = c3;
    return r;
}

// Word stream for one id: counter = (block, id_lo, id_hi, tag), key = seed.
struct WordStream {
    uint32_t k0, k1, id_lo, id_hi, tag, block;
    uint32_t buf[4];
    int pos;
    __device__ uint32_t next()
    {
        if (pos == 4) {
            PhiloxOut o = philox4x32_10(block, id_lo, id_hi, tag, k0, k1);
            buf[0] = o.v[0]; buf[1] = o.v[1]; buf[2] = o.v[2]; buf[3] = o.v[3];
            ++block;
            pos = 0;
        }
        return buf[pos++];
    }
};

#define TAG_EXPANDER 0x41u
#define TAG_NOISE 0x4Eu

// Columns per block of the kernels that write both layouts of A.
#define RL0_COLS 128

// A block's columns [j0, j0 + RL0_COLS) from shared memory (column-major, as in
// rows_cm) to rows_cm (contiguous) and rows_sm (each slot contiguous).
__device__ __forceinline__ void store_columns(const int32_t *sh, int n, int d, int j0, int32_t *rows_cm,
                                              int32_t *rows_sm)
{
    const int cols = min(RL0_COLS, n - j0);
    for (int e = threadIdx.x; e < cols * d; e += RL0_COLS) rows_cm[(int64_t)j0 * d + e] = sh[e];
    if ((int)threadIdx.x < cols)
        for (int s = 0; s < d; ++s) rows_sm[(int64_t)s * n + j0 + threadIdx.x] = sh[threadIdx.x * d + s];
}

// Column j: draw words, map each to [0, m) by Lemire's multiply-shift with
// rejection (exactly uniform), keep the first d distinct values, ascending.  A
// word is inserted into the sorted slots as it comes (DMAX compares in
// registers: a dynamically indexed array lived in local memory).  Both layouts
// are written here: n = 2^22, d = 7: 207 + 88 us (drawing, then slot-major from
// rows_cm) -> 114 us.
template <int DMAX>
__global__ void __launch_bounds__(RL0_COLS) k_make_expander(int n, int m, int d, uint32_t k0, uint32_t k1,
                                                            int32_t *rows_cm, int32_t *rows_sm, int *err)
{
    __shared__ int32_t sh[RL0_COLS * DMAX];
    const int j0 = blockIdx.x * RL0_COLS, j = j0 + threadIdx.x;
    if (j < n) {
        WordStream ws{k0, k1, (uint32_t)j, 0u, TAG_EXPANDER, 0u, {0, 0, 0, 0}, 4};
        int32_t col[DMAX];
#pragma unroll
        for (int q = 0; q < DMAX; ++q) col[q] = 0x7fffffff;
        const uint32_t um = (uint32_t)m;
        const uint32_t thresh = (0u - um) % um;
        int got = 0;
        const int budget = 64 * d + 256;
        for (int draw = 0; draw < budget && got < d; ++draw) {
            const uint64_t prod = (uint64_t)ws.next() * um;
            if ((uint32_t)prod < thresh) continue;  // rejected word
            int32_t c = (int32_t)(prod >> 32);
            bool dup = false;
#pragma unroll
            for (int q = 0; q < DMAX; ++q) dup |= (col[q] == c);
            if (dup) continue;
            ++got;
#pragma unroll
            for (int q = 0; q < DMAX; ++q) {
                const int32_t lo = min(col[q], c);
                c = max(col[q], c);
                col[q] = lo;
            }
        }
        if (got < d) atomicExch(err, 1);
#pragma unroll
        for (int q = 0; q < DMAX; ++q)
            if (q < d) sh[threadIdx.x * d + q] = col[q];
    }
    __syncthreads();
    store_columns(sh, n, d, j0, rows_cm, rows_sm);
}

// Caller rows into both layouts; they must be strictly ascending within a
// column and inside [0, m).  Dynamic shared memory: RL0_COLS d ints.
__global__ void __launch_bounds__(RL0_COLS) k_take_rows(int n, int m, int d, const int32_t *rows, int32_t *rows_cm,
                                                        int32_t *rows_sm, int *bad)
{
    extern __shared__ int32_t sh[];
    const int j0 = blockIdx.x * RL0_COLS, cols = min(RL0_COLS, n - j0);
    for (int e = threadIdx.x; e < cols * d; e += RL0_COLS) sh[e] = rows[(int64_t)j0 * d + e];
    __syncthreads();
    if ((int)threadIdx.x < cols) {
        int32_t prev = -1;
        for (int q = 0; q < d; ++q) {
            const int32_t v = sh[threadIdx.x * d + q];
            if (v <= prev || v >= m) { atomicExch(bad, 1); break; }
            prev = v;
        }
    }
    store_columns(sh, n, d, j0, rows_cm, rows_sm);
}

// ---------------------------------------------------------------------------
// CSR of A^T, columns ascending within a row: a stable two-level sort of the
// entries (in column order) by row.  Rows are split into NB buckets of RB
// consecutive rows.
//   count      tile t (RL0_CSR_TILE entries): its entries per bucket
//   scan       per bucket over the tiles, then over the buckets
//   partition  each tile sorts its entries by bucket in shared memory and writes
//              every bucket's run to its place, packed (row in bucket, column)
//   rows       one CTA per bucket sorts its entries by row in shared memory and
//              writes them, and the bucket's row pointers, in order
// Both sorts are stable counting sorts: a warp takes consecutive entries, 32 at a
// time, and ranks equal keys by __match_any_sync.  Global memory only sees runs: a
// 4-byte store per entry to a place of its own runs at some 65 G stores/s (L2
// merges partial sectors), which is what a counter per row, in global or in
// shared memory, comes down to.  n = 2^22, m = 41943, d = 7: 1230 -> 610 us.
// ---------------------------------------------------------------------------
#define RL0_CSR_TILE 8192
#define RL0_CSR_NT 512                              // threads of the tile kernels
#define RL0_CSR_PER (RL0_CSR_TILE / RL0_CSR_NT)     // entries per thread
#define RL0_CSR_MAX_NB 1024
#define RL0_CSR_ROWS_NT 1024                        // threads of the bucket kernel

struct CsrPlan {
    int nb, rb, ntiles, rbits;                      // buckets, rows per bucket, tiles, bits of a row in its bucket
    int cap;                                        // entries of a bucket that fit shared memory
};

// cnt[bucket ntiles + tile]
__global__ void __launch_bounds__(RL0_CSR_NT) k_csr_count(int nnz, CsrPlan P, const int32_t *rows_cm, int32_t *cnt)
{
    __shared__ int h[RL0_CSR_MAX_NB];
    for (int b = threadIdx.x; b < P.nb; b += RL0_CSR_NT) h[b] = 0;
    __syncthreads();
    const int64_t e0 = (int64_t)blockIdx.x * RL0_CSR_TILE;
#pragma unroll
    for (int u = 0; u < RL0_CSR_PER; ++u) {
        const int64_t e = e0 + u * RL0_CSR_NT + threadIdx.x;
        if (e < nnz) atomicAdd(&h[(unsigned)__ldg(rows_cm + e) / (unsigned)P.rb], 1);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < P.nb; b += RL0_CSR_NT) cnt[(int64_t)b * P.ntiles + blockIdx.x] = h[b];
}

// Inclusive sum over the block of v (256 threads).
__device__ __forceinline__ int block_inclusive256(int v, int *sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) sh[w] = v;
    __syncthreads();
    for (int q = 0; q < w; ++q) v += sh[q];
    __syncthreads();
    return v;
}

// Bucket b's counts to their exclusive prefix over the tiles; tot[b] = its entries.
__global__ void __launch_bounds__(256) k_csr_tile_scan(int ntiles, int32_t *cnt, int32_t *tot)
{
    __shared__ int sh[8], s_run;
    int32_t *c = cnt + (int64_t)blockIdx.x * ntiles;
    int run = 0;
    for (int t0 = 0; t0 < ntiles; t0 += 256) {
        const int t = t0 + threadIdx.x;
        const int v = (t < ntiles) ? c[t] : 0;
        const int incl = block_inclusive256(v, sh);
        if (t < ntiles) c[t] = run + incl - v;
        if (threadIdx.x == 255) s_run = run + incl;
        __syncthreads();
        run = s_run;
        __syncthreads();
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = run;
}

// tot[0 .. nb) to its exclusive prefix, tot[nb] = nnz (one block).
__global__ void __launch_bounds__(256) k_csr_bucket_scan(int nb, int32_t *tot)
{
    __shared__ int sh[8], s_run;
    int run = 0;
    for (int b0 = 0; b0 < nb; b0 += 256) {
        const int b = b0 + threadIdx.x;
        const int v = (b < nb) ? tot[b] : 0;
        const int incl = block_inclusive256(v, sh);
        if (b < nb) tot[b] = run + incl - v;
        if (threadIdx.x == 255) s_run = run + incl;
        __syncthreads();
        run = s_run;
        __syncthreads();
    }
    if (threadIdx.x == 0) tot[nb] = run;
}

// Shared memory: staged entries, their buckets, per-warp bucket counters (16
// bits: a tile holds at most RL0_CSR_TILE), the run's place minus its first
// staged position.
__global__ void __launch_bounds__(RL0_CSR_NT) k_csr_partition(int nnz, int d, CsrPlan P, const int32_t *rows_cm,
                                                              const int32_t *cnt, const int32_t *tot, unsigned *out)
{
    constexpr int NW = RL0_CSR_NT / 32;
    extern __shared__ __align__(16) unsigned char dsm[];
    unsigned *stage = (unsigned *)dsm;
    unsigned short *sb = (unsigned short *)(stage + RL0_CSR_TILE);
    unsigned short *wh = sb + RL0_CSR_TILE;                     // [NW][nb]
    int *delta = (int *)(wh + NW * RL0_CSR_MAX_NB);             // [nb]
    __shared__ int s_scan[NW], s_base;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int i = t; i < NW * P.nb; i += RL0_CSR_NT) wh[i] = 0;
    __syncthreads();
    // warp w: entries e0 + 32 u + lane, u < RL0_CSR_PER, in order
    const int64_t e0 = (int64_t)blockIdx.x * RL0_CSR_TILE + (int64_t)w * 32 * RL0_CSR_PER;
    int row[RL0_CSR_PER];
#pragma unroll
    for (int u = 0; u < RL0_CSR_PER; ++u) {
        const int64_t e = e0 + 32 * u + lane;
        row[u] = (e < nnz) ? __ldg(rows_cm + e) : -1;
    }
    unsigned short *h = wh + w * P.nb;
    unsigned short rank[RL0_CSR_PER];                           // among the warp's entries of the same bucket
#pragma unroll
    for (int u = 0; u < RL0_CSR_PER; ++u) {
        const int b = (row[u] >= 0) ? row[u] / P.rb : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, b);
        const int base = (b >= 0) ? h[b] : 0;
        rank[u] = (unsigned short)(base + __popc(peers & lt));
        __syncwarp();
        if (b >= 0 && (peers & ~lt & ~(1u << lane)) == 0u) h[b] = (unsigned short)(base + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    // per bucket: the warps' counts to their prefix; the buckets' starts in the tile
    if (t == 0) s_base = 0;
    __syncthreads();
    for (int b0 = 0; b0 < P.nb; b0 += RL0_CSR_NT) {
        const int b = b0 + t;
        int total = 0;
        if (b < P.nb)
            for (int q = 0; q < NW; ++q) {
                const int v = wh[q * P.nb + b];
                wh[q * P.nb + b] = (unsigned short)total;
                total += v;
            }
        int incl = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) s_scan[w] = incl;
        __syncthreads();
        int before = s_base;
        for (int q = 0; q < w; ++q) before += s_scan[q];
        const int start = before + incl - total;
        if (b < P.nb) {
            for (int q = 0; q < NW; ++q) wh[q * P.nb + b] = (unsigned short)(wh[q * P.nb + b] + start);
            delta[b] = tot[b] + cnt[(int64_t)b * P.ntiles + blockIdx.x] - start;
        }
        __syncthreads();
        if (t == RL0_CSR_NT - 1) s_base = before + incl;
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < RL0_CSR_PER; ++u) {
        if (row[u] < 0) continue;
        const int b = row[u] / P.rb;
        const int pos = h[b] + rank[u];
        const unsigned col = (unsigned)(e0 + 32 * u + lane) / (unsigned)d;
        stage[pos] = ((unsigned)(row[u] - b * P.rb) << (32 - P.rbits)) | col;
        sb[pos] = (unsigned short)b;
    }
    __syncthreads();
    const int here = (int)min((int64_t)RL0_CSR_TILE, (int64_t)nnz - (int64_t)blockIdx.x * RL0_CSR_TILE);
    for (int p = t; p < here; p += RL0_CSR_NT) out[delta[sb[p]] + p] = stage[p];
}

// Bucket b's entries by row.  Shared memory: cap columns, then [32][rb] counters.
__global__ void __launch_bounds__(RL0_CSR_ROWS_NT) k_csr_rows(int m, CsrPlan P, const unsigned *in, const int32_t *tot,
                                                              int32_t *rowptr, int32_t *colidx)
{
    constexpr int NW = RL0_CSR_ROWS_NT / 32;
    extern __shared__ __align__(16) unsigned char dsm[];
    int32_t *cols = (int32_t *)dsm;
    int *wh = (int *)(cols + P.cap);
    __shared__ int s_scan[NW];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int r0 = blockIdx.x * P.rb, nr = min(P.rb, m - r0);
    const int g0 = tot[blockIdx.x], E = tot[blockIdx.x + 1] - g0;
    const unsigned cmask = (P.rbits >= 32) ? 0u : (0xffffffffu >> P.rbits);
    const bool fits = E <= P.cap;
    for (int i = t; i < NW * P.rb; i += RL0_CSR_ROWS_NT) wh[i] = 0;
    __syncthreads();
    // warp w: entries [w per, (w + 1) per), 32 at a time
    const int per = ((E + NW - 1) / NW + 31) & ~31;
    const int lo = min(E, w * per), hi = min(E, lo + per);
    int *h = wh + w * P.rb;
    for (int p = lo + lane; p < hi; p += 32) atomicAdd(&h[__ldg(in + g0 + p) >> (32 - P.rbits)], 1);
    __syncthreads();
    // rows' starts (rb <= RL0_CSR_ROWS_NT: one row per thread), the warps' prefix within a row
    int total = 0;
    if (t < nr)
        for (int q = 0; q < NW; ++q) {
            const int v = wh[q * P.rb + t];
            wh[q * P.rb + t] = total;
            total += v;
        }
    int incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_scan[w] = incl;
    __syncthreads();
    int start = incl - total;
    for (int q = 0; q < w; ++q) start += s_scan[q];
    if (t < nr) {
        for (int q = 0; q < NW; ++q) wh[q * P.rb + t] += start;
        rowptr[r0 + t] = g0 + start;
        if (r0 + t == m - 1) rowptr[m] = g0 + start + total;
    }
    __syncthreads();
    for (int p0 = lo; p0 < hi; p0 += 32) {
        const int p = p0 + lane;
        const unsigned v = (p < hi) ? __ldg(in + g0 + p) : 0u;
        const int r = (p < hi) ? (int)(v >> (32 - P.rbits)) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, r);
        const int base = (r >= 0) ? h[r] : 0;
        __syncwarp();
        if (r >= 0) {
            const int pos = base + __popc(peers & lt);
            // (a bucket too large for shared memory, from skewed rows, is written entry by entry)
            if (fits) cols[pos] = (int32_t)(v & cmask);
            else colidx[g0 + pos] = (int32_t)(v & cmask);
            if ((peers & ~lt & ~(1u << lane)) == 0u) h[r] = base + __popc(peers);
        }
        __syncwarp();
    }
    if (!fits) return;
    __syncthreads();
    for (int p = t; p < E; p += RL0_CSR_ROWS_NT) colidx[g0 + p] = cols[p];
}

// The same with a global counter per row and an insertion sort per row, for what the
// buckets do not take (rl0_expander_finish): buckets of more than 1024 rows (m above
// a million, or fewer than about two entries per row), more entries per bucket than a
// CTA's shared memory holds beside its counters (n d above 43 million at small m, 20
// million at m = 10^6), or a row in its bucket and a column that do not share 32 bits.
__global__ void k_row_count(int64_t nnz, const int32_t *rows_cm, int32_t *cnt1)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < nnz) atomicAdd(&cnt1[rows_cm[e] + 1], 1);
}

// Exclusive-scan building blocks over int32 (m+1 entries): per-block inclusive
// scan of 1024 values, a scan of the block totals, then the offsets.
__global__ void k_scan_blocks(int len, int32_t *a, int32_t *block_tot)
{
    __shared__ int32_t sh[1024];
    const int i = blockIdx.x * 1024 + threadIdx.x;
    sh[threadIdx.x] = (i < len) ? a[i] : 0;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const int32_t v = (threadIdx.x >= (unsigned)off) ? sh[threadIdx.x - off] : 0;
        __syncthreads();
        sh[threadIdx.x] += v;
        __syncthreads();
    }
    if (i < len) a[i] = sh[threadIdx.x];
    if (threadIdx.x == 1023) block_tot[blockIdx.x] = sh[1023];
}

__global__ void k_scan_totals(int nb, int32_t *tot)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        int32_t run = 0;
        for (int b = 0; b < nb; ++b) { const int32_t v = tot[b]; tot[b] = run; run += v; }
    }
}

__global__ void k_scan_add(int len, int32_t *a, const int32_t *tot)
{
    const int i = blockIdx.x * 1024 + threadIdx.x;
    if (i < len) a[i] += tot[blockIdx.x];
}

__global__ void k_csr_fill(int n, int d, const int32_t *rows_cm, const int32_t *rowptr, int32_t *fill,
                           int32_t *colidx)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)n * d) return;
    const int32_t row = rows_cm[e];
    const int32_t pos = rowptr[row] + atomicAdd(&fill[row], 1);
    colidx[pos] = (int32_t)(e / d);
}

// Sort the columns of every row ascending (insertion sort; rows are short).
__global__ void k_csr_sort(int m, const int32_t *rowptr, int32_t *colidx)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int32_t b = rowptr[i], e = rowptr[i + 1];
    for (int32_t a = b + 1; a < e; ++a) {
        const int32_t v = colidx[a];
        int32_t q = a - 1;
        while (q >= b && colidx[q] > v) { colidx[q + 1] = colidx[q]; --q; }
        colidx[q + 1] = v;
    }
}

// Def. GM items 4 and 6.  Row i: sum of x over its columns (ascending) in FP64,
// plus sigma_n times a Box-Muller deviate of Philox block (0, i, 0, 'N'),
// rounded to FP32 once.
__global__ void k_sketch(int m, const int32_t *rowptr, const int32_t *colidx, const float *x, double sigma_n,
                         uint32_t k0, uint32_t k1, float *y)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    double acc = 0.0;
    for (int32_t p = rowptr[i]; p < rowptr[i + 1]; ++p) acc += (double)x[colidx[p]];
    if (sigma_n > 0.0) {
        PhiloxOut o = philox4x32_10(0u, (uint32_t)i, 0u, TAG_NOISE, k0, k1);
        const double u1 = ((double)o.v[0] + 1.0) / 4294967296.0;
        const double u2 = (double)o.v[1] / 4294967296.0;
        const double z = sqrt(-2.0 * log(u1)) * cos(6.283185307179586476925286766559 * u2);
        acc += sigma_n * z;
    }
    y[i] = (float)acc;
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
int rl0_cuda_err(cudaError_t e)
{
    if (e == cudaSuccess) return RL0_OK;
    if (e == cudaErrorMemoryAllocation) return RL0_ERR_ALLOC;
    return RL0_ERR_CUDA;
}

#define CK(call)                                          \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return rl0_cuda_err(e_);   \
    } while (0)

int rl0_set_device_of(const rl0_expander *A)
{
    int cur = -1;
    CK(cudaGetDevice(&cur));
    if (cur != A->device) CK(cudaSetDevice(A->device));
    return RL0_OK;
}

void rl0_expander_release(rl0_expander *A)
{
    if (!A) return;
    rl0_workspace_free(A);
    cudaFree(A->arena);
    if (A->host_pinned) cudaFreeHost(A->host_pinned);
    delete A;
}

static int check_shape(int64_t n, int64_t m, int d)
{
    if (n < 1 || m < 1 || d < 1 || d > RL0_MAX_D || d > m) return RL0_ERR_INVALID_ARG;
    if (m >= (1LL << 31) || n >= (1LL << 31) || n * (int64_t)d >= (1LL << 31)) return RL0_ERR_INVALID_ARG;
    return RL0_OK;
}

static int alloc_expander(int64_t n, int64_t m, int d, cudaStream_t s, rl0_expander **out)
{
    rl0_expander *A = new (std::nothrow) rl0_expander;
    if (!A) return RL0_ERR_ALLOC;
    std::memset((void *)A, 0, sizeof(*A));
    A->n = n; A->m = m; A->d = d;
    cudaError_t e = cudaGetDevice(&A->device);
    if (e != cudaSuccess) { delete A; return rl0_cuda_err(e); }
    const int rc = rl0_workspace_alloc(A, s);
    if (rc) {
        cudaGetLastError();
        rl0_expander_release(A);
        return rc;
    }
    *out = A;
    return RL0_OK;
}

// CSR of A^T from rows_cm.  The workspace, free until the first decode, lends its
// survivor list (n entries of at least d ints) and its logs.
int rl0_expander_finish(rl0_expander *A, cudaStream_t s)
{
    const int64_t n = A->n, m = A->m;
    const int d = A->d;
    const int64_t nnz = n * d;
    const int len = (int)(m + 1);
    const int nb = (int)rl0_div_up(len, 1024);
    int optin = 0;
    CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, A->device));
    // buckets of at least 2048 entries (at most about 1000 of them); a row in its
    // bucket and a column share 32 bits; a bucket of 1.25 times the mean fits
    CsrPlan P;
    P.nb = (int)std::max<int64_t>(1, std::min<int64_t>({nnz / 2048, 1000, m}));
    P.rb = (int)rl0_div_up(m, P.nb);
    P.nb = (int)rl0_div_up(m, P.rb);
    P.ntiles = (int)rl0_div_up(nnz, RL0_CSR_TILE);
    P.rbits = 1;
    while ((1 << P.rbits) < P.rb) ++P.rbits;
    int cbits = 1;
    while (((int64_t)1 << cbits) < n) ++cbits;
    const int64_t hist = (int64_t)(RL0_CSR_ROWS_NT / 32) * P.rb * 4, room = ((int64_t)optin - 1024 - hist) / 4;
    const size_t cnt_bytes = (size_t)P.nb * P.ntiles * 4 + (size_t)(P.nb + 1) * 4;
    const int64_t want = nnz / P.nb + nnz / P.nb / 4 + 1024;
    if (P.rb <= RL0_CSR_ROWS_NT && P.rbits + cbits <= 32 && want <= room && cnt_bytes <= A->ws.log_bytes) {
        P.cap = (int)want;
        int32_t *cnt = (int32_t *)A->ws.ulog, *tot = cnt + (size_t)P.nb * P.ntiles;
        unsigned *pairs = (unsigned *)A->ws.res_list;
        const int part_smem = 4 * RL0_CSR_TILE + 2 * RL0_CSR_TILE + 2 * (RL0_CSR_NT / 32) * RL0_CSR_MAX_NB +
                              4 * RL0_CSR_MAX_NB;
        const int rows_smem = 4 * P.cap + (int)hist;
        CK(cudaFuncSetAttribute(k_csr_partition, cudaFuncAttributeMaxDynamicSharedMemorySize, part_smem));
        CK(cudaFuncSetAttribute(k_csr_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024));
        k_csr_count<<<P.ntiles, RL0_CSR_NT, 0, s>>>((int)nnz, P, A->rows_cm, cnt);
        k_csr_tile_scan<<<P.nb, 256, 0, s>>>(P.ntiles, cnt, tot);
        k_csr_bucket_scan<<<1, 256, 0, s>>>(P.nb, tot);
        k_csr_partition<<<P.ntiles, RL0_CSR_NT, part_smem, s>>>((int)nnz, d, P, A->rows_cm, cnt, tot, pairs);
        k_csr_rows<<<P.nb, RL0_CSR_ROWS_NT, rows_smem, s>>>((int)m, P, pairs, tot, A->rowptr, A->colidx);
    } else {
        int32_t *fill = nullptr, *tot = nullptr;
        CK(cudaMallocAsync(&tot, (size_t)nb * 4, s));
        CK(cudaMallocAsync(&fill, (size_t)m * 4, s));
        CK(cudaMemsetAsync(A->rowptr, 0, (size_t)(m + 1) * 4, s));
        k_row_count<<<rl0_div_up(nnz, 256), 256, 0, s>>>(nnz, A->rows_cm, A->rowptr);
        k_scan_blocks<<<nb, 1024, 0, s>>>(len, A->rowptr, tot);
        k_scan_totals<<<1, 32, 0, s>>>(nb, tot);
        k_scan_add<<<nb, 1024, 0, s>>>(len, A->rowptr, tot);
        CK(cudaMemsetAsync(fill, 0, (size_t)m * 4, s));
        k_csr_fill<<<rl0_div_up(nnz, 256), 256, 0, s>>>((int)n, d, A->rows_cm, A->rowptr, fill, A->colidx);
        k_csr_sort<<<rl0_div_up(m, 128), 128, 0, s>>>((int)m, A->rowptr, A->colidx);
        CK(cudaFreeAsync(fill, s));
        CK(cudaFreeAsync(tot, s));
    }
    CK(cudaGetLastError());
    return RL0_OK;
}

extern "C" int rl0_make_expander(int64_t n, int64_t m, int d, uint64_t seed, void *cuda_stream,
                                 rl0_expander **out)
{
    if (!out) return RL0_ERR_INVALID_ARG;
    *out = nullptr;
    int rc = check_shape(n, m, d);
    if (rc) return rc;
    rl0_expander *A = nullptr;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    rc = alloc_expander(n, m, d, s, &A);
    if (rc) return rc;
    int err = 0;
    do {
        if (cudaMemsetAsync(A->dev_flag, 0, 4, s) != cudaSuccess) { err = RL0_ERR_CUDA; break; }
#define RL0_MK(D) k_make_expander<D><<<rl0_div_up(n, RL0_COLS), RL0_COLS, 0, s>>>((int)n, (int)m, d, (uint32_t)seed, \
                                                        (uint32_t)(seed >> 32), A->rows_cm, A->rows_sm, A->dev_flag)
        if (d <= 8) RL0_MK(8);
        else if (d <= 16) RL0_MK(16);
        else RL0_MK(32);
#undef RL0_MK
        // (a column that ran out of draws holds INT_MAX: nothing may index with it)
        int flag = 0;
        if (cudaMemcpyAsync(&flag, A->dev_flag, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) { err = RL0_ERR_CUDA; break; }
        if (flag) { err = RL0_ERR_INVALID_ARG; break; }
        err = rl0_expander_finish(A, s);
        if (!err) err = rl0_cuda_err(cudaStreamSynchronize(s));
    } while (0);
    if (err) { cudaGetLastError(); rl0_expander_release(A); return err; }
    *out = A;
    return RL0_OK;
}

extern "C" int rl0_expander_from_rows(int64_t n, int64_t m, int d, const int32_t *rows_dev, void *cuda_stream,
                                      rl0_expander **out)
{
    if (!out || !rows_dev) return RL0_ERR_INVALID_ARG;
    *out = nullptr;
    int rc = check_shape(n, m, d);
    if (rc) return rc;
    rl0_expander *A = nullptr;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    rc = alloc_expander(n, m, d, s, &A);
    if (rc) return rc;
    int err = 0;
    do {
        if (cudaMemsetAsync(A->dev_flag, 0, 4, s) != cudaSuccess) { err = RL0_ERR_CUDA; break; }
        k_take_rows<<<rl0_div_up(n, RL0_COLS), RL0_COLS, RL0_COLS * d * 4, s>>>((int)n, (int)m, d, rows_dev, A->rows_cm,
                                                                                A->rows_sm, A->dev_flag);
        int flag = 0;
        if (cudaMemcpyAsync(&flag, A->dev_flag, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) { err = RL0_ERR_CUDA; break; }
        if (flag) { err = RL0_ERR_INVALID_A; break; }
        err = rl0_expander_finish(A, s);
        if (!err) err = rl0_cuda_err(cudaStreamSynchronize(s));
    } while (0);
    if (err) { cudaGetLastError(); rl0_expander_release(A); return err; }
    *out = A;
    return RL0_OK;
}

extern "C" int rl0_expander_rows(const rl0_expander *A, int32_t *rows_dev, void *cuda_stream)
{
    if (!A || !rows_dev) return RL0_ERR_INVALID_ARG;
    int rc = rl0_set_device_of(A);
    if (rc) return rc;
    CK(cudaMemcpyAsync(rows_dev, A->rows_cm, (size_t)A->n * A->d * 4, cudaMemcpyDeviceToDevice,
                       (cudaStream_t)cuda_stream));
    return RL0_OK;
}

extern "C" int rl0_expander_shape(const rl0_expander *A, int64_t *n, int64_t *m, int *d)
{
    if (!A) return RL0_ERR_INVALID_ARG;
    if (n) *n = A->n;
    if (m) *m = A->m;
    if (d) *d = A->d;
    return RL0_OK;
}

extern "C" void rl0_free_expander(rl0_expander *A)
{
    if (!A) return;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(A->device);
    cudaDeviceSynchronize();
    rl0_expander_release(A);
    if (prev >= 0) cudaSetDevice(prev);
}

extern "C" int rl0_sketch(const rl0_expander *A, const float *x_dev, double sigma_n, uint64_t noise_seed,
                          float *y_dev, void *cuda_stream)
{
    if (!A || !x_dev || !y_dev || !(sigma_n >= 0.0)) return RL0_ERR_INVALID_ARG;
    int rc = rl0_set_device_of(A);
    if (rc) return rc;
    k_sketch<<<rl0_div_up(A->m, 256), 256, 0, (cudaStream_t)cuda_stream>>>(
        (int)A->m, A->rowptr, A->colidx, x_dev, sigma_n, (uint32_t)noise_seed, (uint32_t)(noise_seed >> 32), y_dev);
    CK(cudaGetLastError());
    return RL0_OK;
}

extern "C" const char *rl0_strerror(int code)
{
    switch (code) {
    case RL0_OK: return "success";
    case RL0_ERR_INVALID_ARG: return "invalid argument";
    case RL0_ERR_CUDA: return "CUDA runtime error";
    case RL0_ERR_ALLOC: return "allocation failed";
    case RL0_ERR_TIMEOUT: return "a bounded device wait gave up";
    case RL0_ERR_UNSUPPORTED: return "unsupported request";
    case RL0_ERR_INVALID_A: return "invalid expander rows (range, order or duplicates)";
    case RL0_ERR_INVALID_Y: return "y_hat holds NaN or Inf";
    case RL0_ERR_TOO_LARGE: return "instance larger than the static workspace (n <= 65536, m <= 32768)";
    default: return "unknown error";
    }
}
