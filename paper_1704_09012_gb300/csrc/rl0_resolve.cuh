// rl0_resolve.cuh -- the second half of a round's column score (arXiv
// 1704.09012, Algorithm 2, the loop over j in [n] and i in N(j)): a CTA takes a
// batch of the columns its bound could not rule out, tests their candidate
// anchors exactly and commits the columns that pass.  Shared by both column
// kernels (rl0_column_res.cu, rl0_column_l2.cu).  Not part of the ABI.
#pragma once

#include <type_traits>

#include "rl0_common.cuh"
#include "rl0_device.cuh"
#include "rl0_mma.cuh"
#include "rl0_round.cuh"

// A CTA's state across the batches of one round.
struct ColState {
    Series pe;
    unsigned long long bar;             // completion of the bulk copies (resident codes)
    int count, last;                    // columns listed so far; scratch of the last-CTA test
    unsigned total, ubase, fbase;
    int dn;                             // this CTA's change of the nonzero count
    int next_event;                     // looking ahead: the first later round in which a column passes
    unsigned nnz0;                      // |supp x_hat| at the round's start
};

// Scratch of one batch of NT listed columns and their candidate items (at
// most DMAX each).
template <int DMAX, int NT, bool LEARNED = false>
struct ResScratch {
    float r[DMAX][NT];                   // FP32 residuals of the batch's columns
    float nz[NT], rhs[NT];
    unsigned off[NT];                    // first item of each column
    unsigned short it_e[NT * DMAX];      // item -> column in the batch
    unsigned char it_s[NT * DMAX];       // item -> slot (descending within a column)
    unsigned char it_ok[NT * DMAX];
    float it_w[NT * DMAX];
    float it_sc[NT * DMAX];              // n_e - n_z of the item
    // learned scorer: features of the items that pass the exact tests (compact, NT
    // items at a time; by feature, the pitch keeps a tile's eight rows times four
    // feature pairs on different banks; f14 = f15 = 0 are not held), their items, and the network
    float feat[RL0_NFEAT - 2][LEARNED ? NT + 4 : 1];
    unsigned short fidx[LEARNED ? NT : 1];
    std::conditional_t<LEARNED, MlpPacked, int> mlp;
    float q[NT][DMAX];                   // q_e of (item, slot l), NT items at a time
    unsigned wsum[NT / 32];
    int nf;
};

// Exclusive prefix over the CTA of v (NT threads, all of them call it);
// *total (shared) gets the sum.  wsum: NT / 32 shared words.
template <int NT>
__device__ __forceinline__ unsigned cta_exclusive_scan(unsigned v, unsigned *wsum, unsigned *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const unsigned w = (lane < NT / 32) ? wsum[lane] : 0u;
        unsigned wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        if (lane < NT / 32) wsum[lane] = wi - w;
        if (lane == 31) *total = wi;
    }
    __syncthreads();
    const unsigned r = wsum[warp] + incl - v;
    __syncthreads();
    return r;
}

// One batch: thread t holds listed column j (when act) with its candidate
// slots cm, x_j and the (r, p_z) of its rows in v; rows(rid) gives the column's
// row ids.  ta_look: the anchors to test (th.ta, or the sweep's last t_a when
// the pass looks ahead; those below th.ta only report the round that makes
// them anchors).  net: the learned scorer's network, in shared memory.  Every thread
// of the CTA calls it; the scratch is free again when it returns.  The arithmetic is eval_anchor's, in its order.
template <int DMAX, bool IND, int NT, bool LEARNED, class Rows>
__device__ __forceinline__ void resolve_batch(const KArgs &a, const DecodeCtx *ctx, const RoundThr &th, float ta_look,
                                              int round, int d, int rule, float alpha, int32_t *passed, ResScratch<DMAX, NT, LEARNED> &R,
                                              ColState &S, bool act, int j, unsigned cm, float old, const float2 *v,
                                              Rows rows, const MlpPacked *net = nullptr)
{
    constexpr bool LOOK = !IND && !LEARNED;
    const int tid = threadIdx.x;
    unsigned cand = 0u;
    if (act) {
        float nz = 0.0f, rhs = 0.0f;
#pragma unroll
        for (int s = 0; s < DMAX; ++s) {
            if (s < d) {
                nz += IND ? (fabsf(v[s].x) <= th.tz ? 1.0f : 0.0f) : v[s].y;
                rhs += fabsf(v[s].x);
                // the bound's candidates that are anchors: a superset of the passing
                // anchors, each then tested exactly below
                if (((cm >> s) & 1u) && fabsf(v[s].x) >= (LOOK ? ta_look : th.ta)) cand |= 1u << s;
            }
            R.r[s][tid] = (s < d) ? v[s].x : 0.0f;
        }
        R.nz[tid] = nz;
        R.rhs[tid] = rhs;
    }
    // one item per candidate (column, slot), a column's slots in descending order
    const unsigned nc = (unsigned)__popc(cand);
    const unsigned off = cta_exclusive_scan<NT>(nc, R.wsum, &S.total);
    const unsigned nitems = S.total;
    {
        unsigned c = cand, q = off;
        while (c) {
            const int sl = 31 - __clz(c);
            c &= ~(1u << sl);
            R.it_e[q] = (unsigned short)tid;
            R.it_s[q] = (unsigned char)sl;
            ++q;
        }
    }
    __syncthreads();
    // eval_anchor's arithmetic in two steps, so that an item's d posteriors
    // are evaluated side by side (one per thread) rather than one after
    // another: q_e of every (item, l), then each item's sums in slot order
    for (unsigned k0 = 0; k0 < nitems; k0 += NT) {
        const unsigned kn = min(nitems - k0, (unsigned)NT);
        for (unsigned p = tid; p < kn * (unsigned)d; p += NT) {
            const unsigned kk = p / (unsigned)d, l = p % (unsigned)d;
            const int ee = R.it_e[k0 + kk], sl = R.it_s[k0 + kk];
            const float rs = R.r[sl][ee], rl = R.r[l][ee];
            R.q[kk][l] = IND ? (fabsf(rs - rl) <= th.te ? 1.0f : 0.0f) : series_eval(S.pe, rs - rl);
        }
        __syncthreads();
        for (unsigned kk = tid; kk < kn; kk += NT) {
            const unsigned k = k0 + kk;
            const int ee = R.it_e[k];
            float ne = 0.0f, num = 0.0f;
            for (int l = 0; l < d; ++l) {
                const float rl = R.r[l][ee];
                const float q = R.q[kk][l];
                ne += q;
                num += rl * q;
            }
            const float w = num / ne;
            float lhs = 0.0f;
            for (int l = 0; l < d; ++l) lhs += fabsf(R.r[l][ee] - w);
            if constexpr (LEARNED) {
                // the learned scorer: the l1 test and n_e - n_z >= 1.5 here; the
                // features of the items that pass go to a compact list, whose
                // logits the network takes below
                const bool ok = lhs <= R.rhs[ee] && ne - R.nz[ee] >= ctx->learned_need;
                R.it_ok[k] = ok ? 1 : 0;
                if (ok) {
                    AnchorEval E;
                    E.ne = ne;
                    E.w = w;
                    E.lhs = lhs;
                    float f[RL0_NFEAT];
                    candidate_features(&R.r[0][ee], NT, d, E, R.nz[ee], R.rhs[ee], ctx->inv_sn, th.t, ctx->drho, f);
                    const int p = atomicAdd(&R.nf, 1);
#pragma unroll
                    for (int q = 0; q < RL0_NFEAT - 2; ++q) R.feat[q][p] = f[q];
                    R.fidx[p] = (unsigned short)kk;
                }
            } else {
                R.it_ok[k] = (lhs <= R.rhs[ee] && ne - R.nz[ee] >= alpha) ? 1 : 0;
            }
            R.it_w[k] = w;
            R.it_sc[k] = ne - R.nz[ee];
        }
        __syncthreads();
        if constexpr (LEARNED) {
            // the passing items' logits, 16 per warp on the tensor cores
            const unsigned nf = (unsigned)R.nf;
            for (unsigned t0 = (unsigned)(tid >> 5) * 16u; t0 < nf; t0 += (NT / 32) * 16u) {
                auto f = [&](int r, int i) { return (t0 + r < nf && i < RL0_NFEAT - 2) ? R.feat[i][t0 + r] : 0.0f; };
                float lo, hi;
                warp_mlp_logits16(f, *net, &lo, &hi);
                if ((tid & 3) == 0) {
                    const unsigned gr = (unsigned)((tid & 31) >> 2);
                    if (t0 + gr < nf && !(lo >= ctx->logit_thr)) R.it_ok[k0 + R.fidx[t0 + gr]] = 0;
                    if (t0 + gr + 8 < nf && !(hi >= ctx->logit_thr)) R.it_ok[k0 + R.fidx[t0 + gr + 8]] = 0;
                }
            }
            __syncthreads();
            if (tid == 0) R.nf = 0;                // read again only after the next batch's barriers
        }
    }
    // each column: its first passing item is its highest passing slot (the
    // last passing anchor in row order); with anchor_rule 1 the passing item
    // of largest n_e - n_z, ties to the lower slot (items come highest first)
    int best = -1;
    float bw = 0.0f, bsc = 0.0f, later = 0.0f;
    for (unsigned q = 0; q < nc; ++q)
        if (R.it_ok[off + q]) {
            if (LOOK) {
                const float av = fabsf(R.r[R.it_s[off + q]][tid]);
                if (av < th.ta) {                  // an anchor of a later round
                    later = fmaxf(later, av);
                    continue;
                }
            }
            if (rule == 0) {
                best = R.it_s[off + q];
                bw = R.it_w[off + q];
                break;
            }
            if (best < 0 || R.it_sc[off + q] >= bsc) {
                best = R.it_s[off + q];
                bw = R.it_w[off + q];
                bsc = R.it_sc[off + q];
            }
        }
    if (LOOK && later > 0.0f) atomicMin(&S.next_event, anchor_round(a.thr, round, ctx->nrounds, later));
    const bool pass = best >= 0;
    float nv = old;
    if (pass) {
        nv = old + bw;
        ctx->x[j] = nv;
    }
    if (passed && act) passed[j] = pass ? 1 : 0;
    // a column that became nonzero takes its rows' fresh-bucket slots now,
    // so that those atomics travel with the commit's below
    const bool fresh = pass && old == 0.0f && nv != 0.0f;
    int rid[DMAX], slot[DMAX];
    if (fresh) {
        rows(rid);
        bucket_slots<DMAX>(a, rid, d, slot);
    }
    // the batch's commit: one global atomic per counter
    const unsigned pf = cta_exclusive_scan<NT>((pass ? 0x10000u : 0u) | (fresh ? 1u : 0u), R.wsum, &S.total);
    const unsigned tpf = S.total;
    // entries that became zero; the fresh ones are the scan's low field
    const int ngone = __syncthreads_count(pass && old != 0.0f && nv == 0.0f);
    if (tid == 0) {
        const int nup = (int)(tpf & 0xffffu);
        S.dn += nup - ngone;                       // added to the ticket at the end
        if (ngone) atomicAdd(&a.st->zeroed, (unsigned)ngone);
        const unsigned long long old2 = (tpf != 0u) ? take_upd_list(a.st, tpf >> 16, tpf & 0xffffu) : 0ull;
        S.ubase = (unsigned)(old2 >> 32);
        S.fbase = (unsigned)old2;
    }
    __syncthreads();
    if (pass) {
        UndoEntry u;
        u.j = j;
        u.old = old;
        a.ulog[S.ubase + (pf >> 16)] = u;
    }
    if (fresh) {
        a.list[S.fbase + (pf & 0xffffu)] = j;
        bucket_store<DMAX>(a, j, rid, d, slot);
    }
    __syncthreads();                               // the scratch is reused by the next batch
}
