// rl0_column_l2.cu -- the column score of Robust-l0 (arXiv 1704.09012,
// Algorithm 2, the loop over j in [n] and i in N(j)) with (r, p_z) gathered
// from L2: instances whose residual codes do not fit an SM's shared memory
// (rl0_column_res.cu), and rl0_decode_static, whose workspace holds no codes.
//
// A grid of resident CTAs (res CTAs per SM); CTA b owns the contiguous columns
// [b n / G, (b + 1) n / G) and takes them in chunks of RL0_L2_TILES tiles:
//   stream   one thread per column: its d row ids (coalesced per slot, the next
//            tile's loaded ahead), its d gathers, and the FP32 bound
//            anchor_candidates; a column that survives goes to the CTA's ring in
//            shared memory.  No thread waits on another.
//   resolve  whenever the ring holds a full batch of NT columns (and once at
//            the end), resolve_batch (rl0_resolve.cuh) tests them exactly and
//            commits; its threads are all busy, whatever share of the columns
//            survives.  Other CTAs of the SM stream meanwhile.
//   H_k      in the launch's last CTA, as in the resident-code kernel.
// A queue scored by CTA-wide passes (one candidate slot per column and pass, two
// barriers each) left the warps waiting for one another: 11 of 25 warp-cycles
// per issue at n = 2^22, m = 419 430, d = 7, 19 of 27 with the learned scorer.
// Full batches instead: a whole decode there (39 rounds) 8.62 -> 6.62 ms, a
// learned one (78 rounds) 42.5 -> 33.7 ms, and at n = 2^24, m = 167 772 a round
// 0.71 -> 0.54 ms.  What is left is the gathers: an SM asks L2 for about one
// 32-byte sector per cycle, 0.1 ms for the 29 M of a round at n = 2^22.
#include <algorithm>

#include "rl0_common.cuh"
#include "rl0_device.cuh"
#include "rl0_resolve.cuh"
#include "rl0_round.cuh"

#define RL0_L2_TILES 3                  // tiles per chunk: ring of (tiles + 1) NT entries

namespace {

template <int DMAX> struct L2NT {
    static constexpr int value = DMAX <= 8 ? 256 : (DMAX <= 16 ? 128 : 64);
};

template <int DMAX, int NT, bool LEARNED>
struct L2Shared {
    union {
        ResScratch<DMAX, NT, LEARNED> R;
        struct {
            HkShared hk;
            unsigned suf[NT];
        } h;
    };
    uint2 ring[(RL0_L2_TILES + 1) * NT];   // (column, candidate slots)
    ColState S;
};

// CTAs per SM the registers are bounded for.
template <int DMAX, bool LEARNED> struct L2Occ {
    static constexpr int value = DMAX <= 8 ? (LEARNED ? 3 : 4) : (DMAX <= 16 ? 4 : 6);
};

template <int DMAX, bool IND, bool EXACT, bool LEARNED>
__global__ void __launch_bounds__(L2NT<DMAX>::value, L2Occ<DMAX, LEARNED>::value) k_column_score_l2(KArgs a)
{
    constexpr int NT = L2NT<DMAX>::value;
    constexpr unsigned QC = (RL0_L2_TILES + 1) * NT;
    static_assert((QC & (QC - 1)) == 0, "ring positions wrap by masking");
    extern __shared__ __align__(16) unsigned char dsm[];
    L2Shared<DMAX, NT, LEARNED> &M = *(L2Shared<DMAX, NT, LEARNED> *)dsm;
    ColState &S = M.S;
    DecodeState *st = a.st;
    const DecodeCtx *ctx = a.ctx;
    const int n = a.n, tid = threadIdx.x, lane = tid & 31;
    const int d = EXACT ? DMAX : a.d;
    const int lo = (int)(((long long)blockIdx.x * n) / gridDim.x);
    const int hi = (int)(((long long)(blockIdx.x + 1) * n) / gridDim.x);
    // the first tile's row ids while the previous kernel finishes (A never changes)
    int nxt[DMAX];
#pragma unroll
    for (int s = 0; s < DMAX; ++s) nxt[s] = (s < d && lo + tid < hi) ? __ldg(a.rows_sm + (size_t)s * n + lo + tid) : 0;
    pdl_wait();                                    // the previous rebuild's r, x and state
    const int done = st->done, cur = st->cur, round = st->round, look = st->look;
    const unsigned nnz0 = st->nnz;
    pdl_launch_dependents();
    if (done) return;
    const float2 *rz = cur ? a.rz1 : a.rz0;
    const RoundThr th = a.thr[round];
    if (tid == 0) {
        S.count = 0;
        S.dn = 0;
        S.next_event = 0x7fffffff;
        if (!IND) S.pe = ctx->pe;
        if (LEARNED) M.R.nf = 0;
    }
    const float alpha = ctx->alpha;
    const float need = LEARNED ? (IND ? ctx->learned_need : ctx->learned_need - 1e-3f) : (IND ? alpha : alpha - 1e-3f);
    const float reach = IND ? th.te : ctx->pe.cut, b1 = ctx->pe_b1, c1 = ctx->pe_c1;
    const int rule = ctx->anchor_rule;
    float ta_look = th.ta;
    if (!IND && !LEARNED && look) ta_look = a.thr[ctx->nrounds - 1].ta;
    int32_t *passed = ctx->passed;
    const float *xg = ctx->x;
    __syncthreads();
    unsigned head = 0;                             // ring entries resolved so far
    for (int j0 = lo; j0 < hi;) {
        // ---- stream one chunk
#pragma unroll 1
        for (int c = 0; c < RL0_L2_TILES && j0 < hi; ++c, j0 += NT) {
            int rid[DMAX];
#pragma unroll
            for (int s = 0; s < DMAX; ++s) rid[s] = nxt[s];
            float2 v[DMAX];
            const int j = j0 + tid;
            const bool active = j < hi;
#pragma unroll
            for (int s = 0; s < DMAX; ++s) {
                v[s] = make_float2(0.0f, 0.0f);
                if (s < d && active) v[s] = __ldca(rz + rid[s]);
            }
            {
                const int jn = j + NT;
#pragma unroll
                for (int s = 0; s < DMAX; ++s)
                    if (s < d && jn < hi) nxt[s] = __ldg(a.rows_sm + (size_t)s * n + jn);
            }
            float r[DMAX];
            float nz = 0.0f;
#pragma unroll
            for (int s = 0; s < DMAX; ++s) {
                r[s] = v[s].x;
                if (s < d) nz += IND ? (fabsf(v[s].x) <= th.tz ? 1.0f : 0.0f) : v[s].y;
            }
            const unsigned cm = active ? anchor_candidates<DMAX, IND>(r, d, ta_look, reach, b1, c1, nz, need) : 0u;
            const unsigned m = __ballot_sync(0xffffffffu, cm != 0u);
            if (m) {
                const int leader = __ffs(m) - 1;
                int base = 0;
                if (lane == leader) base = atomicAdd(&S.count, __popc(m));
                base = __shfl_sync(0xffffffffu, base, leader);
                if (cm) M.ring[(unsigned)(base + __popc(m & ((1u << lane) - 1u))) & (QC - 1)] = make_uint2((unsigned)j, cm);
            }
            if (passed && active && !cm) passed[j] = 0;
        }
        __syncthreads();
        // ---- resolve full batches (at the end, the rest too)
        const unsigned cnt = (unsigned)S.count;
        while (cnt - head >= (unsigned)NT || (j0 >= hi && cnt != head)) {
            const unsigned e = head + (unsigned)tid;
            const bool act = e < cnt;
            int j = 0;
            unsigned cm = 0u;
            float old = 0.0f;
            float2 v[DMAX];
            if (act) {
                const uint2 q = M.ring[e & (QC - 1)];
                j = (int)q.x;
                cm = q.y;
                old = __ldca(xg + j);
                const int *ids = a.rows_cm + (size_t)j * d;
#pragma unroll
                for (int s = 0; s < DMAX; ++s) v[s] = (s < d) ? __ldca(rz + __ldg(ids + s)) : make_float2(0.0f, 0.0f);
            }
            auto rows = [&](int *rid) {
                const int *ids = a.rows_cm + (size_t)j * d;
#pragma unroll
                for (int s = 0; s < DMAX; ++s) rid[s] = (s < d) ? __ldg(ids + s) : 0;
            };
            resolve_batch<DMAX, IND, NT, LEARNED>(a, ctx, th, ta_look, round, d, rule, alpha, passed, M.R, S, act, j, cm,
                                                  old, v, rows);
            head += min((unsigned)NT, cnt - head);
        }
    }
    if (!IND && !LEARNED && tid == 0 && S.next_event != 0x7fffffff) atomicMin(&st->next_event, S.next_event);
    last_cta_hk_tick<NT>(a, ctx, M.h.hk, M.h.suf, &S.last, S.dn, nnz0);
}

// Launch shape of a variant: as many CTAs as the SMs hold at once.
template <int DMAX, bool EXACT, bool LEARNED>
void l2_shape(KArgs *a)
{
    constexpr int NT = L2NT<DMAX>::value;
    const unsigned sm = (unsigned)sizeof(L2Shared<DMAX, NT, LEARNED>);
    int nb0 = 0, nb1 = 0;
    a->l2_grid[LEARNED] = 0;
    a->l2_smem[LEARNED] = sm;
    const auto k0 = k_column_score_l2<DMAX, false, EXACT, LEARNED>;
    const auto k1 = k_column_score_l2<DMAX, true, EXACT, LEARNED>;
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (cudaFuncSetAttribute(k0, at, (int)sm) != cudaSuccess || cudaFuncSetAttribute(k1, at, (int)sm) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb0, k0, NT, sm) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb1, k1, NT, sm) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    a->l2_grid[LEARNED] = (int)std::min<long long>((long long)std::min(nb0, nb1) * a->nsm, rl0_div_up(a->n, NT));
}

// Kernel variant of degree d: exact for 6 <= d <= 8, else the smallest DMAX >= d.
template <template <int, bool, bool> class F, bool LEARNED, class... P>
auto l2_variant(int d, P... p)
{
    switch (d) {
    case 6: return F<6, true, LEARNED>::call(p...);
    case 7: return F<7, true, LEARNED>::call(p...);
    case 8: return F<8, true, LEARNED>::call(p...);
    default: break;
    }
    if (d < 6) return F<8, false, LEARNED>::call(p...);
    if (LEARNED || d <= 16) return F<16, false, LEARNED>::call(p...);   // (the learned scorer takes d <= 16)
    return F<LEARNED ? 16 : 32, false, LEARNED>::call(p...);
}

template <int DMAX, bool EXACT, bool LEARNED>
struct L2Shape {
    static bool call(KArgs *a)
    {
        l2_shape<DMAX, EXACT, LEARNED>(a);
        return true;
    }
};

template <int DMAX, bool EXACT, bool LEARNED>
struct L2Launch {
    static bool call(const KArgs *a, int indicator, cudaStream_t s)
    {
        const int grid = a->l2_grid[LEARNED];
        if (grid < 1) return false;
        constexpr int NT = L2NT<DMAX>::value;
        if (indicator) launch_pdl(k_column_score_l2<DMAX, true, EXACT, LEARNED>, grid, NT, a->l2_smem[LEARNED], s, *a);
        else launch_pdl(k_column_score_l2<DMAX, false, EXACT, LEARNED>, grid, NT, a->l2_smem[LEARNED], s, *a);
        return true;
    }
};

}  // namespace

void rl0_l2_setup(KArgs *a)
{
    l2_variant<L2Shape, false>(a->d, a);
    if (a->d <= 16) l2_variant<L2Shape, true>(a->d, a);
}

bool rl0_l2_launch(const KArgs &a, int indicator, int learned, cudaStream_t s)
{
    return learned ? l2_variant<L2Launch, true>(a.d, &a, indicator, s) : l2_variant<L2Launch, false>(a.d, &a, indicator, s);
}
