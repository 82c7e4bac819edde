// local_device.cuh -- the rounds of a peel (Algorithm 2, Sec. 4.1, with
// Algorithms 3 and 4) by one CTA on a live sub-graph whose vertex state is in
// shared memory: the tail of a single peel (peel.cu) and the later rounds of a
// batched graph (batch.cu).
//
// tw[p] is the peeling weight of local vertex p while it is live (>= 0) and
// -i once it left in round i.  The live vertices are grouped in segments of
// 64 with an exact minimum per segment.  A round comes in two forms:
//
//  - Block form, any size: the minima are kept in two buffers by round parity
//    (round i reads its thresholds from one and writes the new minima to the
//    other: recomputed for segments that lose vertices, lowered by atomicMin
//    on every decrement).  The block scans only segments that can hold
//    selected vertices, expands the frontier's arcs with shared-memory
//    atomics, and every warp closes the round and plans the next one itself
//    from the same shared data: two block barriers per round.
//
//  - Warp form, for the minimum-rule rounds of one vertex that make up most of
//    a weighted peel with k(1+eps) < 2: warp 0 runs round after round alone,
//    without barriers, while the others wait.  Its decrements are plain loads
//    and stores, SOLO_ILP chunks of 32 arcs in flight, so no row may hold a head
//    twice: rows that are not known to be strictly increasing (a caller's own) stay
//    with the block form and its atomics.  It hands back to the block at any
//    other round.
//
// Measured (cycles per round at 1.9 GHz): warp form 2,050 with the arcs in
// shared memory, 3,200 with the graph's own rows in L2; block form of one
// vertex 3,000 and 6,100.  A round of hundreds of vertices: 167,000 -> 89,000
// on the 15,000-vertex DG graph, whose peel went from 1,147 to 914 us; the
// smallest window's call without allocation from 289 to 257 us.
#pragma once
#include "peel_device.cuh"

#define SOLO_ILP 4                   // 32-arc chunks in flight
#define SOLO_ARCS (32 * SOLO_ILP)    // most arcs of a warp-form round
#define SOLO_TRY 2                   // the warp form is tried after this many block-form rounds of one vertex ...
#define SOLO_PAYS 2                  // ... or twice as many as last time, up to SOLO_REST, when it ran fewer
#define SOLO_REST 64                 // rounds than this: a try costs about 1 us (a core with rows of 160 arcs,
                                     // which the warp cannot take: 8.3 ms with a try every second round, 6.8 without)

// Where the sub-graph's arcs are.  LocalArcs: copied out, rows end to end, only
// live heads.  GraphArcs: the whole graph's rows, heads looked up in a map from
// vertex to local id (negative: gone before the sub-graph was taken).
struct LocalArcs {
    // Most segments the warp form looks over (twice a round, alone): with the arcs
    // at hand a weighted block graph's peel takes 1.15 ms with and 1.09 without it at
    // 92 segments, 2.62 and 2.43 at 230; 0.63 and 0.70 at 24.
    static constexpr int kSoloSegs = 64;
    const int *toff;       // [L + 1] first arc of each row, in shared memory
    const int *col;        // local heads ...
    const long long *cw;   // ... and weights (nullptr: 1.0)
    __device__ __forceinline__ void row(int p, unsigned &b, unsigned &e) const {
        b = toff[p];
        e = toff[p + 1];
    }
    __device__ __forceinline__ int head(unsigned x) const { return col[x]; }
    __device__ __forceinline__ int local(int h) const { return h; }
    __device__ __forceinline__ long long weight(unsigned x) const { return cw ? cw[x] : DUPIN_Q_ONE; }
};

struct GraphArcs {
    // (the block's rounds wait twice as long for the graph's rows: 160 windows of
    // 60,000 edges take 2.59 ms with and 2.69 without the warp form above 64 segments)
    static constexpr int kSoloSegs = 0x7fffffff;
    const unsigned *start, *deg;  // [L] each row's first arc and arcs, in shared memory
    const int *col, *hubs;
    const long long *cw;          // nullptr: 1.0
    const long long *map;
    __device__ __forceinline__ void row(int p, unsigned &b, unsigned &e) const {
        b = start[p];
        e = b + deg[p];
    }
    __device__ __forceinline__ int head(unsigned x) const { return arc_head(col[x], hubs); }
    __device__ __forceinline__ int local(int h) const { return (int)map[h]; }
    __device__ __forceinline__ long long weight(unsigned x) const { return cw ? cw[x] : DUPIN_Q_ONE; }
};

struct LocalState {
    long long *tw;       // [whole segments] weights, -1 in the last segment's padding
    long long *segbuf;   // [2 nseg]
    unsigned short *tf;  // [L] frontier
    long long L;
    int nseg;
    long long kD, D, max_rounds;
    int use_min, gpo, lpo;
    int repeats;         // a row may hold a head more than once: no warp form
    long long *tr_f_hi;
    unsigned long long *tr_f_lo;
    long long *tr_size, *tr_peeled;
    long long tr_cap;
};

// what the warp form hands back
struct LocalHand {
    long long round, size, gpo_le, gpo_lt, gm_s, n_min_rule, mins, best_round, best_size;
    unsigned long long f_lo, f_hi, gm_lo, gm_hi, bf_lo, bf_hi;
    int rounds;
};

__device__ __forceinline__ void local_trace(const LocalState &S, const RoundState &st, long long peeled) {
    if (st.round < S.tr_cap) {
        S.tr_f_hi[st.round] = (long long)(unsigned long long)(st.f >> 64);
        S.tr_f_lo[st.round] = (unsigned long long)st.f;
        S.tr_size[st.round] = st.size;
        S.tr_peeled[st.round] = peeled;
    }
}

// Warp 0: minimum-rule rounds of one vertex from st (minimum live weight m,
// segment minima in seg) until a round is anything else; returns how many it
// ran.  m is brought up to date.  The path of a round is kept short: one warp
// alone issues about an instruction every four cycles, so a round costs its
// instructions as much as its loads.
template <bool NARROW, class Arcs>
__device__ __forceinline__ int solo_rounds(const LocalState &S, const Arcs &G, long long *seg, RoundState &st, long long &m) {
    const int lane = threadIdx.x & 31;
    const int nseg = S.nseg;
    long long *tw = S.tw;
    int ran = 0;
    while (st.size > 1 && st.round < S.max_rounds) {
        // the plan: with Algorithms 3 and 4 the general one; the round is this
        // warp's when it takes the minimum rule
        if (S.gpo) {
            RoundState t = st;
            const TailRound R = tail_plan<NARROW>(S.kD, S.D, S.use_min, S.gpo, S.lpo, t, m);
            if (!R.minrule) break;
            st.gm_f = t.gm_f;
            st.gm_s = t.gm_s;
            st.gpo_le = t.gpo_le;
            st.gpo_lt = t.gpo_lt;
        } else {
            const u128 X = NARROW ? (u128)(unsigned long long)st.f * (unsigned long long)S.kD
                                  : mul_u128_u64(st.f, (unsigned long long)S.kD);
            if (!S.use_min || mul_le(m, (unsigned long long)S.D * (unsigned long long)st.size,
                                     (unsigned long long)(X >> 64), (unsigned long long)X))
                break;
        }
        // its segment, and the vertex in it: one of each, or the round is the block's
        int cq = -1, nc = 0;
        for (int q0 = 0; q0 < nseg; q0 += 32) {
            const int q = q0 + lane;
            const unsigned cm = __ballot_sync(0xffffffffu, q < nseg && seg[q] == m);
            if (cm) {
                cq = q0 + __ffs(cm) - 1;
                nc += __popc(cm);
            }
        }
        if (nc != 1) break;
        const longlong2 v = *(const longlong2 *)&tw[(long long)cq * 64 + 2 * lane];
        const unsigned b0 = __ballot_sync(0xffffffffu, v.x == m), b1 = __ballot_sync(0xffffffffu, v.y == m);
        if (__popc(b0) + __popc(b1) != 1) break;
        const int p = cq * 64 + (b0 ? 2 * (__ffs(b0) - 1) : 2 * (__ffs(b1) - 1) + 1);
        unsigned x, hi;
        G.row(p, x, hi);
        if (hi - x > SOLO_ARCS) break;
        const int len = (int)(hi - x);
        x += lane;
        const long long i = st.round + 1;
        if (lane == 0) tw[p] = -i;
        {
            long long t = v.x >= 0 && v.x != m ? v.x : kMaxLL;
            if (v.y >= 0 && v.y != m && v.y < t) t = v.y;
            t = warp_min64(t);
            if (lane == 0) seg[cq] = t;
        }
        __syncwarp();
        {
            int cv[SOLO_ILP];
            long long cc[SOLO_ILP];
#pragma unroll
            for (int u = 0; u < SOLO_ILP; u++) {
                if (32 * u >= len) break;
                const bool in = lane + 32 * u < len;
                cv[u] = in ? G.head(x + 32 * u) : -1;
                cc[u] = in ? G.weight(x + 32 * u) : 0;
            }
#pragma unroll
            for (int u = 0; u < SOLO_ILP; u++) {
                if (32 * u >= len) break;
                if (cv[u] >= 0) cv[u] = G.local(cv[u]);
            }
#pragma unroll
            for (int u = 0; u < SOLO_ILP; u++) {
                if (32 * u >= len) break;
                const int h = cv[u];
                if (h >= 0) {
                    const long long nv = tw[h] - cc[u];
                    if (nv + cc[u] >= 0) {  // live; the row's heads are distinct: no other lane has this one
                        tw[h] = nv;
                        if (nv < seg[h >> 6]) atomicMin(&seg[h >> 6], nv);
                    }
                }
            }
        }
        // close: one vertex has no arc to itself
        st.f -= (unsigned long long)m;
        st.size--;
        st.round = i;
        st.n_min_rule++;
        __syncwarp();
        m = kMaxLL;
        for (int q = lane; q < nseg; q += 32) {
            const long long sm = seg[q];
            m = sm < m ? sm : m;
        }
        m = warp_min64(m);
        if (frac_gt<NARROW>(st.f, st.size, st.bf, st.best_size)) {
            st.bf = st.f;
            st.best_size = st.size;
            st.best_round = i;
        }
        if (lane == 0) local_trace(S, st, 1);
        ran++;
    }
    return ran;
}

// exact minima of the segments [wid, nseg) step NW of tw into seg; returns the
// smallest that this warp found
template <int NT>
__device__ __forceinline__ long long local_minima(const long long *tw, int nseg, long long *seg) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long all = kMaxLL;
    for (int q = wid; q < nseg; q += NT / 32) {
        const longlong2 v = *(const longlong2 *)&tw[(long long)q * TAIL_SEG + 2 * lane];
        long long m = kMaxLL;
        if (v.x >= 0) m = v.x;
        if (v.y >= 0 && v.y < m) m = v.y;
        m = warp_min64(m);
        if (lane == 0) seg[q] = m;
        all = m < all ? m : all;
    }
    return all;
}

// All rounds from st to the empty set (or an error, returned).  The segment
// minima of the next round are in the buffer of its parity.  The best prefix
// and the trace are kept by the last warp (its select covers the fewest
// segments): st's best is right in its threads only.
// NARROW: f < 2^62 and the best f < 2^64, so every sum a round forms (at most
// 2f) fits 64 bits; the sums then take 64-bit adds and 32-bit warp reductions,
// the products 64 x 64 -> 128-bit multiplies.
template <int NT, bool NARROW, class Arcs>
__device__ __forceinline__ int local_rounds(const LocalState &S, const Arcs &G, RoundState &st, TailAcc<NT / 32> *s_acc, unsigned *s_rows,
                                            LocalHand *s_hand) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nseg = S.nseg;
    long long *tw = S.tw;
    long long *segbuf = S.segbuf;
    unsigned short *tf = S.tf;
    long long mins_all = seg_global_min(segbuf + ((st.round + 1) & 1) * nseg, nseg);
    TailRound R = tail_plan<NARROW>(S.kD, S.D, S.use_min, S.gpo, S.lpo, st, mins_all);
    // block-form rounds of one vertex in a row; how many before a try of the warp form
    int ones = 0, need = S.repeats || nseg > Arcs::kSoloSegs ? 0x7fffffff : SOLO_TRY;
    while (!R.done) {
        if (R.i > S.max_rounds) return DUPIN_ERR_NO_PROGRESS;
        if (ones >= need && R.minrule) {
            ones = 0;
            const int b0 = (int)(R.i & 1);
            if (tid == (NW - 1) * 32) {
                s_hand->best_round = st.best_round;
                s_hand->best_size = st.best_size;
                s_hand->bf_lo = (unsigned long long)st.bf;
                s_hand->bf_hi = (unsigned long long)(st.bf >> 64);
            }
            __syncthreads();
            if (wid == 0) {
                st.best_round = s_hand->best_round;
                st.best_size = s_hand->best_size;
                st.bf = mk128(s_hand->bf_lo, s_hand->bf_hi);
                long long m = mins_all;
                const int ran = solo_rounds<NARROW>(S, G, segbuf + b0 * nseg, st, m);
                if (lane == 0) {
                    s_hand->round = st.round;
                    s_hand->size = st.size;
                    s_hand->f_lo = (unsigned long long)st.f;
                    s_hand->f_hi = (unsigned long long)(st.f >> 64);
                    s_hand->gpo_le = st.gpo_le;
                    s_hand->gpo_lt = st.gpo_lt;
                    s_hand->gm_lo = (unsigned long long)st.gm_f;
                    s_hand->gm_hi = (unsigned long long)(st.gm_f >> 64);
                    s_hand->gm_s = st.gm_s;
                    s_hand->n_min_rule = st.n_min_rule;
                    s_hand->mins = m;
                    s_hand->rounds = ran;
                    s_hand->best_round = st.best_round;
                    s_hand->best_size = st.best_size;
                    s_hand->bf_lo = (unsigned long long)st.bf;
                    s_hand->bf_hi = (unsigned long long)(st.bf >> 64);
                    s_acc[0].F = 0;
                    s_acc[1].F = 0;
                }
            }
            __syncthreads();
            st.round = s_hand->round;
            st.size = s_hand->size;
            st.f = mk128(s_hand->f_lo, s_hand->f_hi);
            st.gpo_le = s_hand->gpo_le;
            st.gpo_lt = s_hand->gpo_lt;
            st.gm_f = mk128(s_hand->gm_lo, s_hand->gm_hi);
            st.gm_s = s_hand->gm_s;
            st.n_min_rule = s_hand->n_min_rule;
            st.best_round = s_hand->best_round;
            st.best_size = s_hand->best_size;
            st.bf = mk128(s_hand->bf_lo, s_hand->bf_hi);
            mins_all = s_hand->mins;
            need = s_hand->rounds >= SOLO_PAYS ? SOLO_TRY : need < SOLO_REST ? 2 * need : SOLO_REST;
            const bool odd = s_hand->rounds & 1;  // the minima move to the next round's buffer
            if (odd)
                for (int q = tid; q < nseg; q += NT) segbuf[(b0 ^ 1) * nseg + q] = segbuf[b0 * nseg + q];
            __syncthreads();
            R = tail_plan<NARROW>(S.kD, S.D, S.use_min, S.gpo, S.lpo, st, mins_all);
            if (R.done || R.i > S.max_rounds) continue;
        }
        const long long i = R.i;
        const long long *cur = segbuf + (i & 1) * nseg;  // minima at the start of round i
        long long *nxt = segbuf + ((i + 1) & 1) * nseg;  // minima after round i
        TailAcc<NW> &acc = s_acc[i & 1];
        // ---- select: lanes test segments in parallel; a candidate segment
        // is then scanned by its warp (two vertices per lane)
        unsigned long long wlo = 0, whi = 0;
        long long mins = kMaxLL;  // new minimum over the segments this lane looked at
        for (int q0 = wid * 32; q0 < nseg; q0 += NT) {
            const int q = q0 + lane;
            const long long sm = q < nseg ? cur[q] : kMaxLL;
            if (q < nseg) nxt[q] = sm;
            const bool cand = seg_candidate(sm, R);
            if (!cand) mins = sm < mins ? sm : mins;  // untouched by the select
            unsigned cm = __ballot_sync(0xffffffffu, cand);
            __syncwarp();
            while (cm) {
                const int qq = q0 + __ffs(cm) - 1;
                cm &= cm - 1;
                const long long p = (long long)qq * TAIL_SEG + 2 * lane;
                const longlong2 v = *(const longlong2 *)&tw[p];
                bool s0, s1;
                if (R.minrule) {
                    s0 = v.x >= 0 && v.x <= R.minw;
                    s1 = v.y >= 0 && v.y <= R.minw;
                } else {
                    s0 = v.x >= 0 && (v.x <= R.gle || mul_le(v.x, R.Y, R.Xhi, R.Xlo));
                    s1 = v.y >= 0 && (v.y <= R.gle || mul_le(v.y, R.Y, R.Xhi, R.Xlo));
                }
                long long m = kMaxLL;  // the segment's minimum over its survivors
                if (v.x >= 0 && !s0) m = v.x;
                if (v.y >= 0 && !s1 && v.y < m) m = v.y;
                m = warp_min64(m);
                if (lane == 0) {
                    nxt[qq] = m;
                    mins = m < mins ? m : mins;
                }
                const unsigned b0 = __ballot_sync(0xffffffffu, s0), b1 = __ballot_sync(0xffffffffu, s1);
                if (b0 | b1) {
                    unsigned base = 0;
                    if (lane == 0) base = atomicAdd(&acc.F, (unsigned)(__popc(b0) + __popc(b1)));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    const unsigned lt = (1u << lane) - 1u;
                    unsigned slot = base + __popc(b0 & lt) + __popc(b1 & lt);
                    if (s0) {
                        tw[p] = -i;
                        if (NARROW) wlo += (unsigned long long)v.x;
                        else add128(wlo, whi, (unsigned long long)v.x, 0);
                        tf[slot++] = (unsigned short)p;
                    }
                    if (s1) {
                        tw[p + 1] = -i;
                        if (NARROW) wlo += (unsigned long long)v.y;
                        else add128(wlo, whi, (unsigned long long)v.y, 0);
                        tf[slot] = (unsigned short)(p + 1);
                    }
                }
            }
        }
        // the select's sums and minimum stay in registers: they are reduced
        // with the expand's after it, off the path to the first barrier
        __syncthreads();
        // round i+1's counter was last read in round i-1: reset it now
        if (tid == 0) s_acc[(i + 1) & 1].F = 0;
        const int F = (int)acc.F;
        // ---- expand
        unsigned long long ilo = 0, ihi = 0;
        long long mind = kMaxLL;
        if (F <= TAIL_FAST) {
            // the frontier's arcs in chunks of 32 consecutive arcs of one
            // vertex: chunk c goes to warp c % NW, TAIL_ILP of a warp's
            // chunks in flight at once; the walk is the same in every lane
            // (broadcast shared loads, no divergence)
            int e = 0;
            unsigned cbase = 0, c = wid, a0 = 0, a1 = 0;
            if (F > 0) G.row(tf[0], a0, a1);
            while (e < F) {
                int cv[TAIL_ILP];
                long long cc[TAIL_ILP];
                int got = 0;
#pragma unroll
                for (int u = 0; u < TAIL_ILP; u++) {
                    cv[u] = -1;
                    while (e < F && c >= cbase + ((a1 - a0 + 31) >> 5)) {
                        cbase += (a1 - a0 + 31) >> 5;
                        e++;
                        if (e < F) G.row(tf[e], a0, a1);
                    }
                    if (e < F) {
                        const unsigned x = a0 + (c - cbase) * 32 + lane;
                        if (x < a1) {
                            cv[u] = G.head(x);
                            cc[u] = G.weight(x);
                        }
                        c += NW;
                        got++;
                    }
                }
#pragma unroll
                for (int u = 0; u < TAIL_ILP; u++) {
                    if (u >= got) break;
                    if (cv[u] >= 0) cv[u] = G.local(cv[u]);
                }
#pragma unroll
                for (int u = 0; u < TAIL_ILP; u++) {
                    if (u >= got) break;
                    const int v = cv[u];
                    const long long c2 = cc[u];
                    if (v < 0) continue;
                    const long long wv = tw[v];
                    if (wv >= 0) {
                        const long long nv = (long long)atomicAdd((unsigned long long *)&tw[v], (unsigned long long)(-c2)) - c2;
                        if (nv < nxt[v / TAIL_SEG]) atomicMin(&nxt[v / TAIL_SEG], nv);  // minima only fall here
                        mind = nv < mind ? nv : mind;
                    } else if (wv == -i) {
                        if (NARROW) ilo += (unsigned long long)c2;
                        else add128(ilo, ihi, (unsigned long long)c2, 0);
                    }
                }
            }
        } else {
            // Many vertices: each warp takes 32 rows at a time and spreads their
            // arcs over its lanes, without block barriers; decrements return
            // nothing, and the segments' minima are found anew by a pass over
            // the weights (a returning atomic and a minimum per arc cost more).
            unsigned *rs = s_rows + 64 * wid, *rb = rs + 32;
            for (int g0 = 32 * wid; g0 < F; g0 += NT) {
                unsigned b = 0, e = 0;
                if (g0 + lane < F) G.row(tf[g0 + lane], b, e);
                unsigned incl = e - b;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned o = __shfl_up_sync(0xffffffffu, incl, d);
                    if (lane >= d) incl += o;
                }
                rs[lane] = b;
                rb[lane] = incl - (e - b);
                const unsigned tot = __shfl_sync(0xffffffffu, incl, 31);
                __syncwarp();
                for (unsigned x0 = lane; x0 - lane < tot; x0 += 32 * TAIL_ILP) {
                    int cv[TAIL_ILP];
                    long long cc[TAIL_ILP];
#pragma unroll
                    for (int u = 0; u < TAIL_ILP; u++) {
                        const unsigned x = x0 + 32 * u;
                        int t = 0;  // the last row that starts at or before x
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1)
                            if (rb[t + step] <= x) t += step;
                        cv[u] = -1;
                        if (x < tot) {
                            const unsigned pos = rs[t] + (x - rb[t]);
                            cv[u] = G.head(pos);
                            cc[u] = G.weight(pos);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < TAIL_ILP; u++)
                        if (cv[u] >= 0) cv[u] = G.local(cv[u]);
#pragma unroll
                    for (int u = 0; u < TAIL_ILP; u++) {
                        if (cv[u] < 0) continue;
                        const long long wv = tw[cv[u]];
                        if (wv >= 0) {
                            atomicAdd((unsigned long long *)&tw[cv[u]], (unsigned long long)(-cc[u]));
                        } else if (wv == -i) {
                            if (NARROW) ilo += (unsigned long long)cc[u];
                            else add128(ilo, ihi, (unsigned long long)cc[u], 0);
                        }
                    }
                }
                __syncwarp();
            }
            __syncthreads();
            mins = local_minima<NT>(tw, nseg, nxt);
        }
        if (NARROW) {
            if (__any_sync(0xffffffffu, wlo != 0)) wlo = warp_sum64_redux(wlo);
            if (__any_sync(0xffffffffu, ilo != 0)) ilo = warp_sum64_redux(ilo);
        } else {
            if (__any_sync(0xffffffffu, (wlo | whi) != 0)) warp_sum128(wlo, whi);
            if (__any_sync(0xffffffffu, (ilo | ihi) != 0)) warp_sum128(ilo, ihi);
        }
        mins = warp_min64(mind < mins ? mind : mins);
        if (lane == 0) {
            acc.wlo[wid] = wlo;
            acc.whi[wid] = whi;
            acc.ilo[wid] = ilo;
            acc.ihi[wid] = ihi;
            acc.mins[wid] = mins;
        }
        __syncthreads();
        // ---- every warp: close round i and plan round i + 1 (same values everywhere)
        u128 wsel, internal;
        tail_acc_sum<NW, NARROW>(acc, wsel, internal, mins_all);
        st.f = st.f - (wsel - (internal >> 1));
        st.size -= F;
        st.round = i;
        st.n_min_rule += R.minrule ? 1 : 0;
        if (wid == NW - 1 && st.size > 0 && frac_gt<NARROW>(st.f, st.size, st.bf, st.best_size)) {
            st.bf = st.f;
            st.best_size = st.size;
            st.best_round = i;
        }
        if (tid == (NW - 1) * 32) local_trace(S, st, F);
        if (F == 0) return DUPIN_ERR_NO_PROGRESS;  // cannot happen (Lemma 4.2 / minimum rule); stop instead of spinning
        ones = F == 1 ? ones + 1 : 0;
        R = tail_plan<NARROW>(S.kD, S.D, S.use_min, S.gpo, S.lpo, st, mins_all);
    }
    return DUPIN_OK;
}

// bytes of shared memory the state of L vertices takes (tw, segbuf, the rows'
// bounds, tf): 'row' bytes per vertex for the bounds
__host__ __device__ __forceinline__ long long local_bytes(long long L, int row) {
    const long long nseg = (L + TAIL_SEG - 1) / TAIL_SEG;
    return (8 * nseg * TAIL_SEG + 16 * nseg + row * (L + 1) + 2 * L + 15) & ~15LL;
}

// the arrays of S for L vertices from 'smem' on; returns the rows' bounds
__device__ __forceinline__ unsigned *local_layout(LocalState &S, unsigned char *smem, long long L, int row) {
    const int nseg = (int)((L + TAIL_SEG - 1) / TAIL_SEG);
    const long long LP = (long long)nseg * TAIL_SEG;
    S.L = L;
    S.nseg = nseg;
    S.tw = (long long *)smem;
    S.segbuf = (long long *)(smem + 8 * LP);
    S.tf = (unsigned short *)(smem + 8 * LP + 16 * nseg + row * (L + 1));
    return (unsigned *)(smem + 8 * LP + 16 * nseg);
}

// Copies the arcs into shared memory where they fit behind the state (rounds
// then wait for no L2).  No barrier at the end.
template <int NT>
__device__ __forceinline__ void local_stage(LocalArcs &G, unsigned char *smem, long long at, long long bytes, long long arcs) {
    if (arcs <= 0 || at + arcs * (G.cw ? 12 : 4) > bytes) return;
    long long *cw = (long long *)(smem + at);
    int *col = (int *)(cw + (G.cw ? arcs : 0));
    for (long long x = threadIdx.x; x < arcs; x += NT) {
        col[x] = G.col[x];
        if (G.cw) cw[x] = G.cw[x];
    }
    G.col = col;
    if (G.cw) G.cw = cw;
}
