// dense.cu -- the tail of a peel (Algorithm 2, Sec. 4.1, with Algorithms 3 and
// 4 of Sec. 5) on a dense matrix of the live sub-graph's weights, over a
// thread-block cluster of C CTAs (16 where the device allows it, else 8).
//
// On a skewed graph the grid-wide rounds leave a small, dense core (R-MAT
// scale 22: 9,100 vertices, 15% of all pairs joined), and with k(1+eps) < 2
// the thousands of rounds left take one or a few vertices each by the minimum
// rule.  Such a round is bound by its chain of latencies alone.  The sparse
// cluster tail (cluster.cu) needs a group lookup, a gather of heads and
// weights, returning shared-memory atomics, segment minima and a rescan of a
// segment for every removed vertex.  Here row u of an L x L matrix holds
// c_uv for every live v (0 where there is no edge), local vertex v belongs to
// one thread of one CTA for the whole tail, its weight stays in that thread's
// registers, and a round is: load this thread's part of row u, subtract, find
// the minimum.  No atomics, no lists, no gathers.
//
// Layout: CTA r owns the columns [r S, (r + 1) S), S a multiple of 16, thread t
// the G columns from G t on (4, 8 or 16), so a row's part is read in wide
// coalesced pieces.  An element is c_uv without the zero bits that all of the graph's weights end in
// (found when it is loaded), in 1, 4 or 8 bytes as the largest needs: 1 for DG
// and for whole-number weights, 4 for Fraudar's (below 1.0 in Q32.32).
// Rounds by the minimum rule:
//   - every CTA knows the cluster's minimum weight and the vertices at it
//     from the results of round i-1; the loads of the first such row are
//     issued before the round is even closed and planned, so that arithmetic
//     runs while they are in flight; every warp keeps the rows of its lightest
//     vertices prefetched in L2;
//   - each thread subtracts, and each warp finds its minimum and the vertices
//     at it and pushes them into every CTA's inbox, one asynchronous 16-byte
//     shared-memory store per CTA completing on the receiver's mbarrier: the
//     round's only meeting point, no block barrier.
// Other rounds (and ties longer than a record) select in registers, list
// the selected columns per CTA and exchange the lists through distributed
// shared memory around a cluster barrier.
// All arithmetic is exact integer arithmetic, identical to the other tails'.
//
// Measured (2,070 MHz): a round takes 1.01 us on R-MAT scale 24 FD (12,400
// vertices, 4-byte elements; the sparse cluster tail 4.4 us): about 320 cycles
// from the results to the row's loads, 600 for the loads (the plan runs under
// them), 180 to subtract, 360 to the warp's minimum, 600 for the exchange.
// R-MAT scale 24, FD and DG in one call: 70.3 -> 38.5 ms; R-MAT scale 21, DW
// with local trims: 18.8 -> 6.6 ms.  The tail takes over whenever the matrix
// fits the arc buffer it replaces, at any density: its round costs the same on
// a sparse core, where the sparse tail's is still over 3 us.
//
// Inboxes are double-buffered by round parity: a warp pushes round i+2's
// record only after it has received every warp's of round i+1, and a warp
// sends that after its last read of round i's.  A wait that gives up (a lost
// push: cannot happen) records an error and ends its warp; the others then
// miss its pushes and end the same way, and no barrier waits for an exited
// thread.
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <mutex>
#include <string>

#include "cluster_device.cuh"
#include "dupin_internal.h"
#include "peel_device.cuh"

#define DN_TIES 3  // vertices at a warp's minimum that its record takes
#define DN_MAXC 16
#define DN_WARPS (DN_THREADS / 32)
#define DN_RECS (DN_MAXC * DN_WARPS)  // records of a round: one per warp of the cluster
#define DN_AHEAD 4  // rows of a warp's lightest vertices kept prefetched into L2

namespace {

// One warp's results of a round in every CTA's inbox, one 16-byte store ...
struct __align__(16) DnRec {
    long long mn;               // minimum weight of its live vertices (kMaxLL: none)
    unsigned short cnt;         // its live vertices at that weight ...
    unsigned short c[DN_TIES];  // ... by column in the CTA's slice, when cnt <= DN_TIES
};
// ... and another when the round removed several vertices (one vertex has no
// arc to itself): the sum of c over its pairs inside U_i
struct __align__(16) DnIn {
    unsigned long long lo, hi;
};

struct DnSel {
    unsigned cnt, pad;
    unsigned long long w_lo, w_hi;
};

struct DnShared {
    DnRec rec[2][DN_RECS];
    DnIn in[2][DN_RECS];
    DnSel sel[2][DN_MAXC];
    unsigned long long mb[2];
    unsigned long long wlo[DN_WARPS], whi[DN_WARPS];
    unsigned F;
    unsigned short tie[DN_WARPS][4];
    unsigned rm[DN_WARPS][DN_RECS * DN_TIES];  // a warp's list of the vertices a round removes
    unsigned short list[DN_MAX_SLICE];         // a general round's selected columns of this CTA
};

// G neighbouring elements of a row as 32-bit words, loaded 16 bytes at a time
// where there are as many.
template <class E, int G>
struct RowPart {
    static constexpr int NW = G * (int)sizeof(E) / 4;
    unsigned x[NW];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < NW; k++) x[k] = 0;
    }
    __device__ __forceinline__ void load(const E *p) {
        if (NW == 1) {
            x[0] = __ldg((const unsigned *)p);
        } else if (NW == 2) {
            const uint2 v = __ldg((const uint2 *)p);
            x[0] = v.x;
            x[NW > 1 ? 1 : 0] = v.y;
        } else {
#pragma unroll
            for (int k = 0; k + 3 < NW; k += 4) {
                const uint4 v = __ldg((const uint4 *)p + k / 4);
                x[k] = v.x;
                x[k + 1] = v.y;
                x[k + 2] = v.z;
                x[k + 3] = v.w;
            }
        }
    }
    // element b's bits (sizeof(E) <= 4), or its two words
    __device__ __forceinline__ unsigned word(int b) const {
        if (sizeof(E) == 1) return (x[b >> 2] >> (8 * (b & 3))) & 0xffu;
        return x[b];
    }
    __device__ __forceinline__ unsigned long long wide(int b) const {
        return ((unsigned long long)x[2 * b + 1] << 32) | x[2 * b];
    }
};

// a removed vertex's weight in a narrow body (f < 2^62): above any live one,
// and still so after all its later decrements (below 2^62 in sum)
#define DN_GONE (1ll << 62)

// E: matrix element; G: neighbouring columns per thread; NARROW: f < 2^62 and
// the best f < 2^64 at the start (64-bit sums, see the one-CTA tail); HI: the
// weights' low 32 bits are all zero.
template <class E, int G, bool NARROW, bool HI>
__device__ __forceinline__ void dense_body(const PeelArgs &A, const unsigned S_, DnShared &S) {
    constexpr int NT = DN_THREADS, NW = NT / 32;
    constexpr int ROWS = G * (int)sizeof(E) < 64 ? 4 : 2;  // rows in flight
    typedef RowPart<E, G> Part;
    PeelCtl *ctl = A.ctl;
    const unsigned C = cl_size(), r = cl_rank();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const long long L = ctl->live_len;
    const int *live = ctl->live_sel ? A.live1 : A.live0;
    const unsigned c0 = r * S_;        // first column of this CTA
    const unsigned col0 = G * tid;     // first of this thread's, in the slice
    const size_t pitch = (size_t)C * S_;
    const unsigned scale = 1u << (HI ? A.dshift - 32 : A.dshift);
    const E *D = (const E *)A.dmat + c0 + col0;  // this thread's part of row 0
    int *pr = A.pr;

    long long v[G];  // the negated weights: a decrement is one multiply-add
    int gid[G];
    unsigned am = 0, um = 0, pf = 0;  // live columns, columns removed in this round, columns whose rows are prefetched
#pragma unroll
    for (int b = 0; b < G; b++) {
        v[b] = -kMaxLL;
        gid[b] = 0;
        if (col0 < S_ && (long long)(c0 + col0 + b) < L) {
            gid[b] = live[c0 + col0 + b];
            v[b] = -A.w[gid[b]];
            am |= 1u << b;
        }
    }
    RoundState st;  // identical in every thread of every CTA (the best prefix in one warp only)
    st.round = ctl->round;
    st.size = ctl->size;
    st.f = mk128(ctl->f_lo, ctl->f_hi);
    st.best_round = ctl->best_round;
    st.best_size = ctl->best_size;
    st.bf = mk128(ctl->bf_lo, ctl->bf_hi);
    st.gpo_le = ctl->gpo_le;
    st.gpo_lt = ctl->gpo_lt;
    st.gm_f = 0;
    st.gm_s = 0;
    st.n_min_rule = ctl->n_min_rule;
    st.scan = ctl->scan_volume;

    // where lane o pushes: this warp's record in CTA o's inbox, its second part
    // and CTA o's mbarrier, by parity
    uint32_t to[2] = {0, 0}, ti[2] = {0, 0}, tb[2] = {0, 0};
    if (lane < (int)C) {
#pragma unroll
        for (int p = 0; p < 2; p++) {
            to[p] = cl_map(&S.rec[p][r * NW + wid], lane);
            ti[p] = cl_map(&S.in[p][r * NW + wid], lane);
            tb[p] = cl_map(&S.mb[p], lane);
        }
    }
    bool bad = false;  // this warp's wait gave up
    unsigned phase = 0;
    auto wait_results = [&](int pb) {
        if (!mb_try_wait(&S.mb[pb], (phase >> pb) & 1)) {
            const long long t0 = clock64();
            while (!mb_try_wait(&S.mb[pb], (phase >> pb) & 1)) {
                if (clock64() - t0 > (1ll << 32)) {  // a lost push: cannot happen; give up rather than hang
                    bad = true;
                    break;
                }
            }
        }
        bad = __any_sync(0xffffffffu, bad);
        phase ^= 1u << pb;
    };
    // the largest of the columns in 'mask' (negated weights; -kMaxLL: none)
    auto most = [&](unsigned mask, bool all) -> long long {
        long long t[G];
#pragma unroll
        for (int b = 0; b < G; b++) t[b] = all || ((mask >> b) & 1) ? v[b] : -kMaxLL;
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1)
#pragma unroll
            for (int b = 0; b < d; b++) t[b] = t[b + d] > t[b] ? t[b + d] : t[b];
        return t[0];
    };
    // This warp's minimum, its vertices at it and the round's internal sum,
    // pushed into every CTA's inbox (buffer pb).  No block barrier: a round's
    // only meeting point is the mbarrier that all of the cluster's records
    // complete.
    auto publish = [&](int pb, bool internal, unsigned long long il, unsigned long long ih) {
        if (tid == 32) mb_arrive_expect_tx(&S.mb[pb], C * NW * (internal ? 32u : 16u));
        long long wm = warp_min64(-most(am, NARROW));
        if (NARROW && wm >= DN_GONE) wm = kMaxLL;
        unsigned eq = 0;  // this thread's columns at it
#pragma unroll
        for (int b = 0; b < G; b++)
            if (v[b] == -wm) eq |= 1u << b;
        eq &= am;
        const unsigned bal = __ballot_sync(0xffffffffu, eq != 0);
        unsigned x = ((col0 + __ffs(eq) - 1) << 16) | 1u, y = 0;  // one vertex at it: the record's count and first column
        if ((eq & (eq - 1)) != 0) x = 0;
        x = __shfl_sync(0xffffffffu, x, (__ffs(bal) - 1) & 31);
        if (bal == 0) {
            x = 0;
        } else if ((bal & (bal - 1)) != 0 || x == 0) {  // ties inside the warp
            unsigned cnt = 0;
#pragma unroll
            for (int b = 0; b < G; b++) {
                const unsigned bb = __ballot_sync(0xffffffffu, (eq >> b) & 1);
                const unsigned slot = cnt + __popc(bb & lt);
                if (((eq >> b) & 1) && slot < DN_TIES) S.tie[wid][slot] = (unsigned short)(col0 + b);
                cnt += __popc(bb);
            }
            __syncwarp();
            x = (cnt > 0xffffu ? 0xffffu : cnt) | ((unsigned)S.tie[wid][0] << 16);
            y = S.tie[wid][1] | ((unsigned)S.tie[wid][2] << 16);  // entries past cnt: stale, unread
            __syncwarp();
        }
        if (internal) {
            if (NARROW) {
                il = warp_sum64_redux(il);
            } else {
                warp_sum128(il, ih);
                il = __shfl_sync(0xffffffffu, il, 0);
                ih = __shfl_sync(0xffffffffu, ih, 0);
            }
        }
        if (lane < (int)C) {
            cl_st_async_v4(pb ? to[1] : to[0], pb ? tb[1] : tb[0], (unsigned)wm, (unsigned)((unsigned long long)wm >> 32), x, y);
            if (internal)
                cl_st_async_v4(pb ? ti[1] : ti[0], pb ? tb[1] : tb[0], (unsigned)il, (unsigned)(il >> 32), (unsigned)ih,
                               (unsigned)(ih >> 32));
        }
        // While the results travel: the rows of this warp's lightest vertices
        // into L2 (each warp keeps DN_AHEAD of them there, and always its
        // lightest), so that a removed vertex's row rarely comes from DRAM.
        if (wm != kMaxLL) {
            const unsigned out = __reduce_add_sync(0xffffffffu, (unsigned)__popc(pf & am));
            const long long z = most(am & ~pf, false);
            const long long zm = warp_min64(-z);
            if (zm != kMaxLL && (out < DN_AHEAD || zm == wm)) {
                const unsigned who = __ballot_sync(0xffffffffu, -z == zm);
                if (lane == __ffs(who) - 1) {
                    unsigned xb = 0;
#pragma unroll
                    for (int b = 0; b < G; b++)
                        if ((((am & ~pf) >> b) & 1) && v[b] == z) xb = b;
                    pf |= 1u << xb;
                    const size_t id = c0 + col0 + xb;
                    prefetch_l2(A.dmat, (unsigned long long)L * pitch * sizeof(E), id * pitch * sizeof(E), pitch * sizeof(E));
                }
            }
        }
    };

    // this thread's part of a row; one with no column that needs it is left out
    auto load_row = [&](unsigned id, Part &a) {
        a.clear();
        if ((am | um) != 0) a.load(D + (size_t)id * pitch);
    };
    // the cluster's results (buffer pb), read by every warp alike
    long long Mn = kMaxLL;        // minimum live weight
    unsigned nat0 = 0, nat1 = 0;  // vertices at it in records lane and lane + 32
    uint2 cc0, cc1;               // those records' counts and columns
    bool over = false;            // a list longer than its record
    unsigned total = 0;           // vertices at it (when !over)
    unsigned id0 = 0;             // the first of them
    Part a0;                      // its row
    const unsigned nrec = C * NW;
    const unsigned base0 = (unsigned)(lane / NW) * S_, base1 = (unsigned)((lane + 32) / NW) * S_;
    auto results = [&](int pb, bool internal, unsigned long long &Il, unsigned long long &Ih) {
        const uint4 p = *(const uint4 *)&S.rec[pb][lane];
        const uint4 q = *(const uint4 *)&S.rec[pb][lane + 32 < (int)nrec ? lane + 32 : lane];
        const long long m0 = (long long)(((unsigned long long)p.y << 32) | p.x);
        const long long m1 = (long long)(((unsigned long long)q.y << 32) | q.x);
        cc0 = make_uint2(p.z, p.w);
        cc1 = make_uint2(q.z, q.w);
        Mn = warp_min64(m1 < m0 ? m1 : m0);
        const bool is0 = m0 == Mn && Mn != kMaxLL;
        const bool is1 = m1 == Mn && Mn != kMaxLL && lane + 32 < (int)nrec;
        const unsigned at = __ballot_sync(0xffffffffu, is0 || is1);
        if (at) {
            const unsigned id = is0 ? base0 + (p.z >> 16) : base1 + (q.z >> 16);
            id0 = __shfl_sync(0xffffffffu, id, __ffs(at) - 1);
            load_row(id0, a0);  // in flight while the round closes
        }
        nat0 = is0 ? p.z & 0xffffu : 0;
        nat1 = is1 ? q.z & 0xffffu : 0;
        over = __any_sync(0xffffffffu, nat0 > DN_TIES || nat1 > DN_TIES);
        total = __reduce_add_sync(0xffffffffu, nat0 + nat1);
        Il = 0;
        Ih = 0;
        if (internal) {
            Il = S.in[pb][lane].lo;
            Ih = S.in[pb][lane].hi;
            if (lane + 32 < (int)nrec) add128(Il, Ih, S.in[pb][lane + 32].lo, S.in[pb][lane + 32].hi);
            if (NARROW) {
                Il = warp_sum64_redux(Il);
            } else {
                warp_sum128(Il, Ih);
                Il = __shfl_sync(0xffffffffu, Il, 0);
                Ih = __shfl_sync(0xffffffffu, Ih, 0);
            }
        }
    };
    // column id leaves in round i: its thread marks it
    auto mark = [&](unsigned id, int i) {
        const unsigned c = id - c0 - col0;
        if (c < G && col0 < S_) {
#pragma unroll
            for (int b = 0; b < G; b++)
                if (c == (unsigned)b) {
                    pr[gid[b]] = i;
                    if (NARROW) v[b] = -kMaxLL;
                }
            am &= ~(1u << c);
            um |= 1u << c;
        }
    };

    if (tid == 0) {
        mb_init(&S.mb[0], 1);
        mb_init(&S.mb[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        S.F = 0;
    }
    __syncthreads();
    cl_sync();  // every CTA's mbarriers are set up before any push
    int err = 0;
    unsigned long long Il, Ih;
    TailRound R;
    bool fast;
    long long noted = st.round;  // the last round in the trace
    unsigned last_un = 0;
    // the best prefix and the trace entry of the last closed round: one warp of
    // one CTA, while a round's results travel
    auto note = [&]() {
        if (r != 0 || wid != NW - 1 || st.round == noted) return;
        noted = st.round;
        if (st.size > 0 && frac_gt<NARROW>(st.f, st.size, st.bf, st.best_size)) {
            st.bf = st.f;
            st.best_size = st.size;
            st.best_round = st.round;
        }
        if (lane == 0 && st.round < A.tr_cap) {
            A.tr_f_hi[st.round] = (long long)(unsigned long long)(st.f >> 64);
            A.tr_f_lo[st.round] = (unsigned long long)st.f;
            A.tr_size[st.round] = st.size;
            A.tr_peeled[st.round] = last_un;
        }
    };
    publish((int)(st.round & 1), false, 0, 0);
    wait_results((int)(st.round & 1));
    if (!bad) results((int)(st.round & 1), false, Il, Ih);
    R = tail_plan<NARROW>(A.kD, A.D, A.use_min, A.gpo, A.lpo, st, Mn);
    fast = R.minrule && !over;
    while (!bad && !R.done) {
        if (R.i > A.max_rounds) {
            err = DUPIN_ERR_NO_PROGRESS;
            break;
        }
        const long long i = R.i;
        const int par = (int)(i & 1);
        unsigned long long Wl, Wh;  // sum of the removed vertices' weights
        unsigned Un;
        unsigned long long ilo = 0, ihi = 0;
        auto apply = [&](const Part &a, bool inside) {
#pragma unroll
            for (int b = 0; b < G; b++) {
                if (!NARROW && !((am >> b) & 1)) continue;
                if (sizeof(E) == 8) {
                    v[b] += (long long)a.wide(b);
                } else if (HI) {
                    const unsigned h = (unsigned)((unsigned long long)v[b] >> 32) + a.word(b) * scale;
                    v[b] = (long long)(((unsigned long long)h << 32) | (unsigned)v[b]);
                } else {
                    v[b] = (long long)((unsigned long long)v[b] + (unsigned long long)a.word(b) * scale);
                }
            }
            if (inside && um) {
#pragma unroll
                for (int b = 0; b < G; b++) {
                    if (!((um >> b) & 1)) continue;
                    const unsigned long long c =
                        sizeof(E) == 8 ? a.wide(b) : ((unsigned long long)a.word(b) * scale) << (HI ? 32 : 0);
                    if (NARROW) ilo += c;
                    else add128(ilo, ihi, c, 0);
                }
            }
        };
        um = 0;
        if (fast) {
            Un = total;
            const u128 W = (u128)(unsigned long long)R.minw * Un;
            Wl = (unsigned long long)W;
            Wh = (unsigned long long)(W >> 64);
            if (Un == 1) {
                mark(id0, (int)i);
                apply(a0, false);
            } else {
                unsigned *rm = S.rm[wid];
                unsigned incl = nat0 + nat1;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned o = __shfl_up_sync(0xffffffffu, incl, d);
                    if (lane >= d) incl += o;
                }
                unsigned at = incl - nat0 - nat1;
                const unsigned c0s[3] = {cc0.x >> 16, cc0.y & 0xffffu, cc0.y >> 16};
                const unsigned c1s[3] = {cc1.x >> 16, cc1.y & 0xffffu, cc1.y >> 16};
#pragma unroll
                for (int k = 0; k < DN_TIES; k++)
                    if ((unsigned)k < nat0) rm[at++] = base0 + c0s[k];
#pragma unroll
                for (int k = 0; k < DN_TIES; k++)
                    if ((unsigned)k < nat1) rm[at++] = base1 + c1s[k];
                __syncwarp();
                Part x[ROWS];
#pragma unroll
                for (int k = 0; k < ROWS; k++)
                    if (1 + k < Un) load_row(rm[1 + k], x[k]);
                for (unsigned e = 0; e < Un; e++) mark(rm[e], (int)i);
                apply(a0, true);
                for (unsigned e = 1; e < Un; e += ROWS) {
#pragma unroll
                    for (int k = 0; k < ROWS; k++)
                        if (e + k < Un) apply(x[k], true);
#pragma unroll
                    for (int k = 0; k < ROWS; k++)
                        if (e + ROWS + k < Un) load_row(rm[e + ROWS + k], x[k]);
                }
                __syncwarp();
            }
        } else {
            // select this thread's columns; list them per CTA
            unsigned long long wlo = 0, whi = 0;
#pragma unroll
            for (int b = 0; b < G; b++) {
                const long long w = -v[b];
                bool s = false;
                if ((am >> b) & 1) s = R.minrule ? w <= R.minw : (w <= R.gle || mul_le(w, R.Y, R.Xhi, R.Xlo));
                const unsigned bal = __ballot_sync(0xffffffffu, s);
                if (!bal) continue;
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(&S.F, (unsigned)__popc(bal));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (s) {
                    S.list[base + __popc(bal & lt)] = (unsigned short)(col0 + b);
                    am &= ~(1u << b);
                    um |= 1u << b;
                    pr[gid[b]] = (int)i;
                    if (NARROW) wlo += (unsigned long long)w;
                    else add128(wlo, whi, (unsigned long long)w, 0);
                    if (NARROW) v[b] = -kMaxLL;
                }
            }
            if (NARROW) wlo = warp_sum64_redux(wlo);
            else warp_sum128(wlo, whi);
            if (lane == 0) {
                S.wlo[wid] = wlo;
                S.whi[wid] = whi;
            }
            __syncthreads();
            if (wid == 0) {
                unsigned long long l = lane < NW ? S.wlo[lane] : 0, h = lane < NW ? S.whi[lane] : 0;
                warp_sum128(l, h);
                l = __shfl_sync(0xffffffffu, l, 0);
                h = __shfl_sync(0xffffffffu, h, 0);
                if (lane < (int)C) {
                    const uint32_t b = cl_map(&S.sel[par][r], lane);
                    cl_st_u32(b + offsetof(DnSel, cnt), S.F);
                    cl_st_u64(b + offsetof(DnSel, w_lo), l);
                    cl_st_u64(b + offsetof(DnSel, w_hi), h);
                }
            }
            cl_sync();  // every CTA's selection and list are visible
            if (tid == 0) S.F = 0;
            const unsigned cq = lane < (int)C ? S.sel[par][lane].cnt : 0;
            Un = __reduce_add_sync(0xffffffffu, cq);
            Wl = lane < (int)C ? S.sel[par][lane].w_lo : 0;
            Wh = lane < (int)C ? S.sel[par][lane].w_hi : 0;
            warp_sum128(Wl, Wh);
            Wl = __shfl_sync(0xffffffffu, Wl, 0);
            Wh = __shfl_sync(0xffffffffu, Wh, 0);
            for (unsigned q = 0; q < C; q++) {
                const unsigned n = __shfl_sync(0xffffffffu, cq, q);
                const uint32_t lq = cl_map(S.list, q);
                for (unsigned e0 = 0; e0 < n; e0 += 32) {
                    const unsigned mine = e0 + lane < n ? q * S_ + cl_ld_u16(lq + 2 * (e0 + lane)) : 0;
                    const unsigned m = n - e0 < 32 ? n - e0 : 32;
                    for (unsigned e = 0; e < m; e += ROWS) {
                        Part x[ROWS];
#pragma unroll
                        for (int k = 0; k < ROWS; k++) {
                            const unsigned id = __shfl_sync(0xffffffffu, mine, (e + k) & 31);
                            if (e + k < m) load_row(id, x[k]);
                        }
#pragma unroll
                        for (int k = 0; k < ROWS; k++)
                            if (e + k < m) apply(x[k], true);
                    }
                }
            }
        }
        const bool internal = Un > 1;  // one vertex has no arc to itself
        publish(par, internal, ilo, ihi);
        note();
        wait_results(par);
        if (bad) break;
        // ---- close round i and plan round i+1 (every warp, same values)
        results(par, internal, Il, Ih);
        if (NARROW) st.f = (u128)((unsigned long long)st.f - (Wl - (Il >> 1)));
        else st.f = st.f - (mk128(Wl, Wh) - (mk128(Il, Ih) >> 1));
        st.scan += st.size;
        st.size -= Un;
        st.round = i;
        st.n_min_rule += R.minrule ? 1 : 0;
        last_un = Un;
        R = tail_plan<NARROW>(A.kD, A.D, A.use_min, A.gpo, A.lpo, st, Mn);
        fast = R.minrule && !over;
        if (Un == 0) R.i = A.max_rounds + 1;  // cannot happen (Lemma 4.2 / minimum rule): leave without progress
    }
    if (bad) {  // this warp leaves for good: no barrier waits for an exited thread
        set_error(ctl, DUPIN_ERR_TIMEOUT);
        return;
    }
    note();
    if (r == 0 && tid == (NW - 1) * 32) {
        if (err) set_error(ctl, err);
        ctl->round = st.round;
        ctl->size = st.size;
        ctl->f_lo = (unsigned long long)st.f;
        ctl->f_hi = (unsigned long long)(st.f >> 64);
        ctl->best_round = st.best_round;
        ctl->best_size = st.best_size;
        ctl->bf_lo = (unsigned long long)st.bf;
        ctl->bf_hi = (unsigned long long)(st.bf >> 64);
        ctl->gpo_le = st.gpo_le;
        ctl->gpo_lt = st.gpo_lt;
        ctl->n_min_rule = st.n_min_rule;
        ctl->scan_volume = st.scan;
        ctl->tail_ctas = (int)C;
    }
    cl_sync();  // no CTA leaves while another may still push to it or read its list
    if (r == 0 && tid == (NW - 1) * 32 && !err) ctl->status = ST_DONE;
}

template <class E, bool HI>
__device__ __forceinline__ void dense_forms(const PeelArgs &A, DnShared &S) {
    const PeelCtl *c = A.ctl;
    const unsigned S_ = (unsigned)dense_slice(c->live_len, A.cl_c);
    const bool narrow = c->f_hi == 0 && c->f_lo < (1ull << 62) && c->bf_hi == 0;
    if (!narrow) dense_body<E, 16, false, HI>(A, S_, S);
    else if (S_ <= 4 * DN_THREADS) dense_body<E, 4, true, HI>(A, S_, S);
    else if (S_ <= 8 * DN_THREADS) dense_body<E, 8, true, HI>(A, S_, S);
    else dense_body<E, 16, true, HI>(A, S_, S);
}

template <class E>
__global__ void __launch_bounds__(DN_THREADS, 1) k_peel_dense(PeelArgs A) {
    __shared__ DnShared S;
    if (A.ctl->status != ST_DENSE || A.ctl->error) return;  // identical in every CTA
    if (sizeof(E) == 8 || A.dshift < 32) dense_forms<E, false>(A, S);
    else dense_forms<E, sizeof(E) != 8>(A, S);
}

// The matrix, cleared: L rows of C S elements, 16 bytes per store (the pitch
// in bytes is a multiple of 16: S is a multiple of 16 elements).
__global__ void k_dense_clear(PeelArgs A) {
    const PeelCtl *c = A.ctl;
    if (c->status != ST_DENSE || c->error) return;
    const long long L = c->live_len;
    const long long bytes = L * A.cl_c * dense_slice(L, A.cl_c) * A.desz;
    const uint4 z = make_uint4(0, 0, 0, 0);
    uint4 *d = (uint4 *)A.dmat;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < bytes / 16; x += (long long)gridDim.x * blockDim.x)
        d[x] = z;
}

// The live arcs of every live vertex's row, written into the matrix: one walk
// over the rows (the sparse tails' builds need two: a count and a fill).
__global__ void __launch_bounds__(BULK_THREADS) k_dense_fill(PeelArgs A) {
    __shared__ WalkShared s_walk;
    __shared__ long long s_k0;
    __shared__ unsigned s_cnt;
    const PeelCtl *c = A.ctl;
    if (c->status != ST_DENSE || c->error) return;
    const long long L = c->live_len;
    const int *live = c->live_sel ? A.live1 : A.live0;
    const long long tot = A.tdeg[L];
    const long long e0 = split_at(tot, blockIdx.x, gridDim.x);
    const long long e1 = split_at(tot, blockIdx.x + 1, gridDim.x);
    if (e0 >= e1) return;
    const long long *tdeg = A.tdeg;
    const long long *rp = A.g.rp;
    if (threadIdx.x < 32) {
        const long long k = warp_search_last_le(tdeg, L, e0);
        if (threadIdx.x == 0) {
            s_k0 = k;
            s_cnt = 0;
        }
    }
    __syncthreads();
    const long long k0 = s_k0;
    const int *col = A.g.col;
    const int *hubs = A.g.hubs;
    const long long *cw = A.g.cw;
    const RankWord *rank = A.rank;
    const size_t pitch = (size_t)A.cl_c * dense_slice(L, A.cl_c);
    unsigned cnt = 0;
    walk_arcs<BULK_THREADS, BUILD_ILP, true>(
        [=](long long k) { return tdeg[k]; }, [=](long long k) { return rp[live[k]]; }, L, e0, e1, k0, s_walk,
        [&](const long long (&k)[BUILD_ILP], const long long (&pos)[BUILD_ILP]) {
            int v[BUILD_ILP], to[BUILD_ILP];
#pragma unroll
            for (int u = 0; u < BUILD_ILP; u++) v[u] = pos[u] >= 0 ? col[pos[u]] : 0;
#pragma unroll
            for (int u = 0; u < BUILD_ILP; u++) {
                if (v[u] < 0) v[u] = hubs[-v[u] - 1];
                if (pos[u] >= 0 && !((rank[v[u] >> 5].live >> (v[u] & 31)) & 1u)) v[u] = -1;
                if (pos[u] < 0) v[u] = -1;
            }
#pragma unroll
            for (int u = 0; u < BUILD_ILP; u++) to[u] = v[u] >= 0 ? A.loc[v[u]] : 0;
#pragma unroll
            for (int u = 0; u < BUILD_ILP; u++) {
                if (v[u] < 0) continue;
                const size_t at = (size_t)k[u] * pitch + (size_t)to[u];
                const unsigned long long q = (unsigned long long)(cw ? cw[pos[u]] : DUPIN_Q_ONE) >> A.dshift;
                if (A.desz == 1) ((unsigned char *)A.dmat)[at] = (unsigned char)q;
                else if (A.desz == 4) ((unsigned *)A.dmat)[at] = (unsigned)q;
                else ((long long *)A.dmat)[at] = (long long)q;
                cnt++;
            }
        });
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_cnt, cnt);
    __syncthreads();
    // the arcs the tail began with: counted here unless the cluster tail was first
    if (threadIdx.x == 0 && !c->handed) atomicAdd((unsigned long long *)&A.ctl->tail_arcs, (unsigned long long)s_cnt);
}

}  // namespace

long long dense_cap(long long bytes, int esz, int C) {
    if (C <= 0) return 0;
    long long lo = 0, hi = (long long)C * DN_MAX_SLICE;
    while (lo < hi) {
        const long long L = (lo + hi + 1) / 2;
        if (L * C * dense_slice(L, C) * esz <= bytes) lo = L;
        else hi = L - 1;
    }
    return lo;
}

int launch_dense_build(const PeelArgs &A, int sms, cudaStream_t s) {
    k_dense_clear<<<sms * 4, 512, 0, s>>>(A);
    k_dense_fill<<<sms * 2, BULK_THREADS, 0, s>>>(A);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DUPIN_OK : dupin_cuda_fail(e, "dense tail build");
}

// One cluster of A.cl_c CTAs (the sparse cluster tail's shape; this kernel
// needs less shared memory).
int launch_dense_tail(const PeelArgs &A, cudaStream_t s) {
    static std::mutex mu;
    static bool done[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return dupin_fail(DUPIN_ERR_CUDA, "device ordinal out of range");
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!done[dev]) {
            for (const void *f : {(const void *)k_peel_dense<long long>, (const void *)k_peel_dense<unsigned>,
                                  (const void *)k_peel_dense<unsigned char>}) {
                cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
                if (e != cudaSuccess) return dupin_cuda_fail(e, "cudaFuncSetAttribute(k_peel_dense)");
            }
            done[dev] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(A.cl_c);
    cfg.blockDim = dim3(DN_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = A.cl_c;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = A.desz == 8   ? cudaLaunchKernelEx(&cfg, k_peel_dense<long long>, A)
                    : A.desz == 4 ? cudaLaunchKernelEx(&cfg, k_peel_dense<unsigned>, A)
                                  : cudaLaunchKernelEx(&cfg, k_peel_dense<unsigned char>, A);
    if (e != cudaSuccess) return dupin_cuda_fail(e, "cluster launch of k_peel_dense");
    return DUPIN_OK;
}
