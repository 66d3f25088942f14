// rl0_column_l2.cu -- the column score of Robust-l0 (arXiv 1704.09012,
// Algorithm 2, the loop over j in [n] and i in N(j)) with (r, p_z) gathered
// from L2: instances whose residual codes do not fit an SM's shared memory
// (rl0_column_res.cu), and rl0_decode_static, whose workspace holds no codes.
//
// d = 6, 7, 8: a grid of resident CTAs; CTA b owns the contiguous columns
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
// barriers each) left the warps waiting for one another: barriers were 8.7 of 25.7
// warp-cycles per issue at n = 2^22, m = 419 430, d = 7, 17 with the learned
// scorer.  Full batches instead: a round there 218 -> 150 us (learned 790 -> 199,
// with the packed network), a whole decode of 39 rounds 8.62 -> 6.59 ms, and at
// n = 2^24, m = 167 772 a round 0.71 -> 0.54 ms.  What is left is the gathers: an
// SM asks L2 for 0.8 32-byte sectors per cycle, 34 M in a round at n = 2^22.
#include <algorithm>
#include <type_traits>

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
    // (column, candidate slots), with the learned scorer in one word, (column - lo) << 8
    // | slots (n d < 2^31 and d >= 6: a CTA of at least 152 has fewer than 2^24 columns).
    // Its three CTAs leave little of the SM's memory to L1: with 68 KB each a decode at
    // n = 2^22, m = 419 430 took 43.8 ms, with 62 KB 32.5.  The analytic kernel has the
    // room and not the register (4.07 ms packed, 3.86 not).
    std::conditional_t<LEARNED, unsigned, uint2> ring[(RL0_L2_TILES + 1) * NT];
    ColState S;
};

// CTAs per SM the registers are bounded for.
template <bool LEARNED> struct L2Occ {
    static constexpr int value = LEARNED ? 3 : 4;
};

template <int DMAX, bool IND, bool LEARNED>
__global__ void __launch_bounds__(L2NT<DMAX>::value, L2Occ<LEARNED>::value) k_column_score_l2(KArgs a)
{
    constexpr int NT = L2NT<DMAX>::value;
    constexpr unsigned QC = (RL0_L2_TILES + 1) * NT;
    static_assert((QC & (QC - 1)) == 0, "ring positions wrap by masking");
    static_assert(DMAX <= 8, "a ring entry holds 8 candidate slots");
    extern __shared__ __align__(16) unsigned char dsm[];
    L2Shared<DMAX, NT, LEARNED> &M = *(L2Shared<DMAX, NT, LEARNED> *)dsm;
    ColState &S = M.S;
    DecodeState *st = a.st;
    const DecodeCtx *ctx = a.ctx;
    const int n = a.n, tid = threadIdx.x, lane = tid & 31;
    constexpr int d = DMAX;
    const int lo = (int)(((long long)blockIdx.x * n) / gridDim.x);
    const int hi = (int)(((long long)(blockIdx.x + 1) * n) / gridDim.x);
    // the first tile's row ids while the previous kernel finishes (A never changes)
    int nxt[DMAX];
#pragma unroll
    for (int s = 0; s < DMAX; ++s) nxt[s] = (lo + tid < hi) ? __ldg(a.rows_sm + (size_t)s * n + lo + tid) : 0;
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
    if constexpr (LEARNED) mlp_pack(M.R.mlp, (const __nv_bfloat16 *)ctx->mlp, tid, NT);   // (read after the barriers below)
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
                if (active) v[s] = __ldca(rz + rid[s]);
            }
            {
                const int jn = j + NT;
#pragma unroll
                for (int s = 0; s < DMAX; ++s)
                    if (jn < hi) nxt[s] = __ldg(a.rows_sm + (size_t)s * n + jn);
            }
            float r[DMAX];
            float nz = 0.0f;
#pragma unroll
            for (int s = 0; s < DMAX; ++s) {
                r[s] = v[s].x;
                nz += IND ? (fabsf(v[s].x) <= th.tz ? 1.0f : 0.0f) : v[s].y;
            }
            const unsigned cm = active ? anchor_candidates<DMAX, IND>(r, d, ta_look, reach, b1, c1, nz, need) : 0u;
            const unsigned m = __ballot_sync(0xffffffffu, cm != 0u);
            if (m) {
                const int leader = __ffs(m) - 1;
                int base = 0;
                if (lane == leader) base = atomicAdd(&S.count, __popc(m));
                base = __shfl_sync(0xffffffffu, base, leader);
                if (cm) {
                    auto &q = M.ring[(unsigned)(base + __popc(m & ((1u << lane) - 1u))) & (QC - 1)];
                    if constexpr (LEARNED) q = ((unsigned)(j - lo) << 8) | cm;
                    else q = make_uint2((unsigned)j, cm);
                }
            }
            if (passed && active && !cm) passed[j] = 0;
        }
        __syncthreads();
        // ---- resolve full batches (at the end, the rest too).  Every thread takes the
        // same count: the next chunk adds to it only after all have read it, also when
        // no batch is resolved (whose barriers would keep the warps together).
        const unsigned cnt = (unsigned)S.count;
        __syncthreads();
        while (cnt - head >= (unsigned)NT || (j0 >= hi && cnt != head)) {
            const unsigned e = head + (unsigned)tid;
            const bool act = e < cnt;
            int j = 0;
            unsigned cm = 0u;
            float old = 0.0f;
            float2 v[DMAX];
            if (act) {
                const auto q = M.ring[e & (QC - 1)];
                if constexpr (LEARNED) {
                    j = lo + (int)(q >> 8);
                    cm = q & 0xffu;
                } else {
                    j = (int)q.x;
                    cm = q.y;
                }
                old = __ldca(xg + j);
                const int *ids = a.rows_cm + (size_t)j * d;
#pragma unroll
                for (int s = 0; s < DMAX; ++s) v[s] = __ldca(rz + __ldg(ids + s));
            }
            auto rows = [&](int *rid) {
                const int *ids = a.rows_cm + (size_t)j * d;
#pragma unroll
                for (int s = 0; s < DMAX; ++s) rid[s] = __ldg(ids + s);
            };
            resolve_batch<DMAX, IND, NT, LEARNED>(a, ctx, th, ta_look, round, d, rule, alpha, passed, M.R, S, act, j, cm,
                                                  old, v, rows, LEARNED ? (const MlpPacked *)&M.R.mlp : nullptr);
            head += min((unsigned)NT, cnt - head);
        }
    }
    if (!IND && !LEARNED && tid == 0 && S.next_event != 0x7fffffff) atomicMin(&st->next_event, S.next_event);
    last_cta_hk_tick<NT>(a, ctx, M.h.hk, M.h.suf, &S.last, S.dn, nnz0);
}

// ---------------------------------------------------------------------------
// Degrees other than 6, 7, 8: one CTA per tile of NT columns.  The general
// variants' columns (up to 16 or 32 slots) take the registers and the shared
// memory that the resolve above needs for its batches: at d = 9, n = 805 348,
// m = 214 919 the resident form took 152 us per round, this one 56 (d = 20: 1864
// and 239).  The candidates are queued in passes, one slot per column and pass,
// highest slot first, and scored by the whole CTA.
// ---------------------------------------------------------------------------
// A 32-bit ticket (a launch here can have more CTAs than the resident kernels' 16-bit
// count takes): the launch's last CTA applies H_k when |supp x'| > k (state read past L1,
// since other CTAs updated it during this launch).  hk and suf are scratch of
// that CTA; *last is a shared flag.
template <int NT>
__device__ __forceinline__ void last_cta_hk(const KArgs &a, const DecodeCtx *ctx, HkShared &hk, unsigned *suf,
                                            int *last)
{
    __syncthreads();
    if (threadIdx.x == 0) *last = (cta_ticket(&a.st->col_done) == gridDim.x - 1u);
    __syncthreads();
    if (!*last) return;
    DecodeState *stw = a.st;
    const unsigned upd = __ldcg(&stw->upd_count);
    const long long nnz = (long long)__ldcg(&stw->nnz) + __ldcg(&stw->nnz_delta);
    if (threadIdx.x == 0) stw->col_done = 0u;
    if (upd == 0 || nnz <= ctx->k || __ldcg(&stw->status) != 0) return;
    cta_hk_select<NT>(a.list, __ldcg(&stw->list_count), ctx->x, ctx->k, a.hkkey, a.dlog, &stw->drop_count, hk, suf);
}

// Column j's outcome: x_j += omega of its chosen anchor (best >= 0), with the
// undo log, the support list and the nonzero count kept in step.  Every lane
// of the warp calls it; the warp's leader takes its undo-log and list slots
// with one atomic (take_upd_list).
__device__ __forceinline__ void commit_column(const KArgs &a, const DecodeCtx *ctx, int j, bool active, int best,
                                              float bw)
{
    const bool pass = best >= 0;
    float old = 0.0f, nv = 0.0f;
    if (pass) {
        float *x = ctx->x;
        old = x[j];
        nv = old + bw;
        x[j] = nv;
    }
    if (ctx->passed && active) ctx->passed[j] = pass ? 1 : 0;
    const int lane = threadIdx.x & 31;
    const unsigned mask = __ballot_sync(0xffffffffu, pass);
    if (mask) {
        const int leader = __ffs(mask) - 1;
        const int dn = __reduce_add_sync(0xffffffffu, pass ? (int)(nv != 0.0f) - (int)(old != 0.0f) : 0);
        const unsigned gone = __popc(__ballot_sync(0xffffffffu, pass && old != 0.0f && nv == 0.0f));
        const bool fresh = pass && old == 0.0f && nv != 0.0f;
        const unsigned fmask = __ballot_sync(0xffffffffu, fresh);
        // d <= 8: a fresh column's row ids and bucket slots, before (and so in
        // flight with) the leader's atomic below
        int rid[8], slot[8];
        const bool early = fresh && a.d <= 8;
        if (early) {
#pragma unroll
            for (int q = 0; q < 8; ++q) rid[q] = (q < a.d) ? __ldg(a.rows_sm + (size_t)q * a.n + j) : 0;
            bucket_slots<8>(a, rid, a.d, slot);
        }
        unsigned base = 0, fbase = 0;
        if (lane == leader) {
            if (dn) atomicAdd(&a.st->nnz_delta, dn);
            if (gone) atomicAdd(&a.st->zeroed, gone);
            const unsigned long long old2 = take_upd_list(a.st, (unsigned)__popc(mask), (unsigned)__popc(fmask));
            base = (unsigned)(old2 >> 32);
            fbase = (unsigned)old2;
        }
        base = __shfl_sync(0xffffffffu, base, leader);
        fbase = __shfl_sync(0xffffffffu, fbase, leader);
        const unsigned below = (1u << lane) - 1u;
        if (pass) {
            UndoEntry e;
            e.j = j;
            e.old = old;
            a.ulog[base + __popc(mask & below)] = e;
        }
        if (early) {
            a.list[fbase + __popc(fmask & below)] = j;
            bucket_store<8>(a, j, rid, a.d, slot);
        } else if (fresh) {
            a.list[fbase + __popc(fmask & below)] = j;
            // into the rebuild's fresh buckets, up to 8 rows at a time
            for (int s0 = 0; s0 < a.d; s0 += 8) {
                int rid[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) rid[q] = (s0 + q < a.d) ? __ldg(a.rows_sm + (size_t)(s0 + q) * a.n + j) : 0;
                bucket_column<8>(a, j, rid, min(8, a.d - s0));
            }
        }
    }
}

// Shared memory of the column kernels.  H_k's scratch (used by the launch's
// last CTA after its tiles) shares the bytes of the candidate queue.
template <int DMAX, int NT, bool LEARNED>
struct ColShared {
    union {
        struct {
            float r[DMAX][NT];                 // residuals of columns with candidates
            float nz[NT], rhs[NT];
            unsigned short q[NT];              // this pass's queue: (column lane << 5) | slot
            float score[NT], w[NT];
            unsigned char ok[NT];
            float f[LEARNED ? RL0_NFEAT : 1][LEARNED ? NT : 1];   // features of the candidates that pass
            unsigned short fq[LEARNED ? NT : 1];                  // their queue positions
        } c;
        struct {
            HkShared hk;
            unsigned suf[NT];
        } h;
    };
    Series pe;
    int nq, nf;
    int last, next_event;
};

template <int DMAX, bool IND, bool LEARNED, int NT>
__device__ __forceinline__ void col_setup(const DecodeCtx *ctx, ColShared<DMAX, NT, LEARNED> &S)
{
    const int tid = threadIdx.x;
    if (tid == 0) {
        S.nq = 0;
        S.nf = 0;
        S.next_event = 0x7fffffff;
        if (!IND) S.pe = ctx->pe;
    }
    // (these shared copies are first read after a barrier of the tile body)
}

// One tile of NT columns starting at j0.  gather(row) returns (r_row, p_z(r_row)).
template <int DMAX, bool IND, bool LEARNED, int NT, class Gather>
__device__ __forceinline__ void score_tile(const KArgs &a, const DecodeCtx *ctx, const RoundThr &th, float ta_look,
                                           int round, int j0, Gather gather, ColShared<DMAX, NT, LEARNED> &S)
{
    const int tid = threadIdx.x;
    const int n = a.n, d = a.d;
    const int j = j0 + tid;
    const bool active = j < n;
    const float alpha = ctx->alpha;

    float r[DMAX];
    float nz = 0.0f, rhs = 0.0f;
#pragma unroll
    for (int s = 0; s < DMAX; ++s) {
        r[s] = 0.0f;
        if (s < d && active) {
            const float2 v = gather(__ldg(a.rows_sm + (size_t)s * n + j));
            r[s] = v.x;
            nz += IND ? (fabsf(v.x) <= th.tz ? 1.0f : 0.0f) : v.y;
            rhs += fabsf(v.x);
        }
    }
    const float need = LEARNED ? (IND ? ctx->learned_need : ctx->learned_need - 1e-3f) : (IND ? alpha : alpha - 1e-3f);
    unsigned cand = active ? anchor_candidates<DMAX, IND>(r, d, ta_look, IND ? th.te : ctx->pe.cut, ctx->pe_b1,
                                                          ctx->pe_c1, nz, need) : 0u;
    if (cand) {
#pragma unroll
        for (int s = 0; s < DMAX; ++s) S.c.r[s][tid] = r[s];
        S.c.nz[tid] = nz;
        S.c.rhs[tid] = rhs;
    }
    int best = -1;
    float bw = 0.0f, bsc = 0.0f, later = 0.0f;
    while (__syncthreads_or(cand != 0u)) {
        int my = -1, ms = 0;
        if (cand) {
            ms = 31 - __clz(cand);                  // highest remaining slot first
            cand &= ~(1u << ms);
            my = atomicAdd(&S.nq, 1);
            S.c.q[my] = (unsigned short)((tid << 5) | ms);
        }
        __syncthreads();
        const int nq = S.nq;
        if (LEARNED) {
            // the learned scorer's logit replaces n_e - n_z >= alpha: each queued
            // candidate's exact l1 test and n_e - n_z >= 1.5 first; the features
            // of those that pass go to a compact list, whose logits the MLP takes
            // 16 per warp on the tensor cores (rl0_mma.cuh: the arithmetic of
            // rl0_mlp_forward); a candidate passes when its logit reaches the
            // threshold
            for (int e = tid; e < nq; e += NT) {
                const int owner = S.c.q[e] >> 5, s = S.c.q[e] & 31;
                const AnchorEval E = eval_anchor<IND>(&S.c.r[0][owner], NT, d, s, th.te, S.pe);
                S.c.ok[e] = 0;
                S.c.score[e] = 0.0f;
                S.c.w[e] = E.w;
                if (E.lhs <= S.c.rhs[owner] && E.ne - S.c.nz[owner] >= ctx->learned_need) {
                    const int p = atomicAdd(&S.nf, 1);
                    float f[RL0_NFEAT];
                    candidate_features(&S.c.r[0][owner], NT, d, E, S.c.nz[owner], S.c.rhs[owner], ctx->inv_sn,
                                       th.t, ctx->drho, f);
#pragma unroll
                    for (int q = 0; q < RL0_NFEAT; ++q) S.c.f[q][p] = f[q];
                    S.c.fq[p] = (unsigned short)e;
                }
            }
            __syncthreads();
            const int nf = S.nf;
            const __nv_bfloat16 *wb = (const __nv_bfloat16 *)ctx->mlp;
            for (int e0 = (tid >> 5) * 16; e0 < nf; e0 += (NT / 32) * 16) {
                auto f = [&](int r, int i) { return (e0 + r < nf) ? S.c.f[i][e0 + r] : 0.0f; };
                float lo, hi;
                warp_mlp_logits16(f, MlpGlobal{wb}, &lo, &hi);
                if ((tid & 3) == 0) {
                    const int gr = (tid & 31) >> 2;
                    if (e0 + gr < nf) {
                        const int e = S.c.fq[e0 + gr];
                        S.c.score[e] = lo;
                        S.c.ok[e] = (lo >= ctx->logit_thr) ? 1 : 0;
                    }
                    if (e0 + gr + 8 < nf) {
                        const int e = S.c.fq[e0 + gr + 8];
                        S.c.score[e] = hi;
                        S.c.ok[e] = (hi >= ctx->logit_thr) ? 1 : 0;
                    }
                }
            }
        } else {
            for (int e = tid; e < nq; e += NT) {
                const int owner = S.c.q[e] >> 5, s = S.c.q[e] & 31;
                float sc, w;
                S.c.ok[e] = score_anchor<IND>(&S.c.r[0][owner], NT, d, s, th.te, S.pe, S.c.nz[owner], S.c.rhs[owner],
                                              alpha, &sc, &w) ? 1 : 0;
                S.c.score[e] = sc;
                S.c.w[e] = w;
            }
        }
        __syncthreads();
        if (my >= 0 && S.c.ok[my]) {
            const float av = fabsf(S.c.r[ms][tid]);
            if (!IND && !LEARNED && av < th.ta) {   // an anchor of a later round (looking ahead)
                later = fmaxf(later, av);
            } else if (ctx->anchor_rule == 0) {            // the first pass from the top is the last passing
                best = ms;                          // anchor in row order: it stands, the rest is moot
                bw = S.c.w[my];
                cand = 0u;
            } else if (best < 0 || S.c.score[my] >= bsc) {   // largest n_e - n_z; slots come highest
                best = ms;                                   // first, so >= leaves ties to the lower row
                bw = S.c.w[my];
                bsc = S.c.score[my];
            }
        }
        if (tid == 0) {
            S.nq = 0;
            S.nf = 0;
        }
    }
    if (!IND && !LEARNED && later > 0.0f) atomicMin(&S.next_event, anchor_round(a.thr, round, ctx->nrounds, later));
    commit_column(a, ctx, j, active, best, bw);
}

template <int DMAX, bool IND, bool LEARNED>
__global__ void __launch_bounds__(L2NT<DMAX>::value) k_column_score_tile(KArgs a)
{
    constexpr int NT = L2NT<DMAX>::value;
    __shared__ ColShared<DMAX, NT, LEARNED> S;
    const DecodeState *st = a.st;
    pdl_wait();                                    // the previous rebuild's r, x and state
    const int done = st->done, cur = st->cur, round = st->round, look = st->look;
    pdl_launch_dependents();
    if (done) return;
    const DecodeCtx *ctx = a.ctx;
    const float2 *rz = cur ? a.rz1 : a.rz0;
    const RoundThr th = a.thr[round];
    float ta_look = th.ta;
    if (!IND && !LEARNED && look) ta_look = a.thr[ctx->nrounds - 1].ta;
    col_setup<DMAX, IND, LEARNED, NT>(ctx, S);
    score_tile<DMAX, IND, LEARNED, NT>(a, ctx, th, ta_look, round, blockIdx.x * NT,
                                       [rz](int row) { return __ldg(rz + row); }, S);
    __syncthreads();
    if (!IND && !LEARNED && threadIdx.x == 0 && S.next_event != 0x7fffffff)
        atomicMin(&a.st->next_event, S.next_event);
    last_cta_hk<NT>(a, ctx, S.h.hk, S.h.suf, &S.last);
}

// Launch shape of a variant: as many CTAs as the SMs hold at once (0 when the device
// refuses it: a decode that needs the variant returns RL0_ERR_CUDA).
template <int DMAX, bool LEARNED>
void l2_shape(KArgs *a)
{
    constexpr int NT = L2NT<DMAX>::value;
    const unsigned sm = (unsigned)sizeof(L2Shared<DMAX, NT, LEARNED>);
    int nb0 = 0, nb1 = 0;
    a->l2_grid[LEARNED] = 0;
    a->l2_smem[LEARNED] = sm;
    const auto k0 = k_column_score_l2<DMAX, false, LEARNED>;
    const auto k1 = k_column_score_l2<DMAX, true, LEARNED>;
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
        if constexpr (EXACT) {
            l2_shape<DMAX, LEARNED>(a);
        } else {
            a->l2_grid[LEARNED] = (int)rl0_div_up(a->n, L2NT<DMAX>::value);
            a->l2_smem[LEARNED] = 0;
        }
        return true;
    }
};

template <int DMAX, bool EXACT, bool LEARNED>
struct L2Launch {
    static int call(const KArgs *a, int indicator, cudaStream_t s)
    {
        const int grid = a->l2_grid[LEARNED];
        if (grid < 1) return RL0_ERR_CUDA;          // the setup could not get the kernel's shape
        constexpr int NT = L2NT<DMAX>::value;
        const unsigned sm = a->l2_smem[LEARNED];
        if constexpr (EXACT) {
            if (indicator) launch_pdl(k_column_score_l2<DMAX, true, LEARNED>, grid, NT, sm, s, *a);
            else launch_pdl(k_column_score_l2<DMAX, false, LEARNED>, grid, NT, sm, s, *a);
        } else {
            if (indicator) launch_pdl(k_column_score_tile<DMAX, true, LEARNED>, grid, NT, sm, s, *a);
            else launch_pdl(k_column_score_tile<DMAX, false, LEARNED>, grid, NT, sm, s, *a);
        }
        return RL0_OK;
    }
};

}  // namespace

void rl0_l2_setup(KArgs *a)
{
    l2_variant<L2Shape, false>(a->d, a);
    if (a->d <= 16) l2_variant<L2Shape, true>(a->d, a);
}

int rl0_l2_launch(const KArgs &a, int indicator, int learned, cudaStream_t s)
{
    return learned ? l2_variant<L2Launch, true>(a.d, &a, indicator, s) : l2_variant<L2Launch, false>(a.d, &a, indicator, s);
}
