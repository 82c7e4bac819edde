// tds.cu -- batch peeling under the clique metrics of Sec. 2.1: TDS
// (triangle density) and kCLiDS (q-clique density).  f(S) = number of
// q-cliques of G[S] (q = 3 for TDS), w_u(S) = the q-cliques of G[S] through
// u, so that removing u lowers f by w_u.  The rounds are Algorithm 2 (Sec.
// 4.1; the paper's k for these metrics is q) with Algorithm 3's tau_max and
// Algorithm 4's trims by flag, exactly as for the other metrics but on plain
// counts (no Q32.32 scale): every comparison is between ratios of integers.
//
// Device state lives in one control block; a round is four launches --
//   select  every live u with w_u <= T leaves: its round is recorded and it
//           joins the round's list;
//   expand  the cliques of G[S_{i-1}] that die, listed once each (below), in
//           two launches by the size of a vertex's candidate set; each lowers
//           f by one and each member outside U_i by one;
//   close   the minimum live weight; the last block closes the round (f, |S|,
//           the trace, the best prefix) and plans the next one: a trim round
//           if some live w < g(S) (Algorithm 4), else a main round (w <=
//           max(tau_max, k(1+eps) g)), or the minimum rule if that threshold
//           selects nobody.
// The host launches rounds in groups (2, 4, 8, ... 32) and reads the control
// block between groups; launches after the peel ends return at once.
//
// Listing.  A clique belongs to its member u of lowest rank = (degree, id); a
// dying one to its removed member of lowest rank.  u's candidates P are its
// neighbours that may be the others: those that outrank u, or in a round the
// ones in S_{i-1} that survive it or outrank u.  The cliques of u are the
// (q-1)-cliques of G[P], and the ones through v in P are the (q-2)-cliques of
// G[P] among v's neighbours: popcounts over ANDed rows of P's adjacency
// matrix in shared memory, so no clique is visited one by one and w is
// updated once per (u, v).  Whether two candidates are adjacent comes from one
// bit of a global matrix over the (at most) CORE_MAX vertices of highest
// degree; outside it the rows themselves are read, or searched where they are
// long.  (A row merge or a leapfrog walk per arc, one warp per u, read hub
// rows of thousands for every arc of a hub.  One peel, k = q: R-MAT scale 15
// TDS 63.4 -> 1.32 ms, scale 13 4-cliques 417 -> 0.87 ms; what is left is bound
// by the latency of the bit lookups and row reads.)
// A warp takes a vertex of at most WARP_P candidates and LONG_ROW arcs, a CTA one of up to
// CTA_P candidates (one SM's shared memory; for triangles, which need no matrix, P
// itself is the limit); larger ones fall back to a depth-first walk over the
// rows.  Rows are sorted (the loader checks it).
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <string>
#include <type_traits>

#include "dupin_internal.h"

namespace {

constexpr int QMAX = DUPIN_CLIQUE_MAX_Q;
constexpr int CORE_MAX = 8192;             // vertices of the adjacency matrix (8 MB)
constexpr int CORE_WORDS = CORE_MAX / 32;  // its row
constexpr int DEG_BINS = 4096;
constexpr int WARP_P = 128;                // candidates of a warp's vertex
constexpr int WARP_STRIDE = WARP_P / 32 + 1;
constexpr int LONG_ROW = 4096;             // a warp reads no longer row for a vertex's candidates
constexpr int READ_ARCS = 192;             // a candidate's row is read when it has no more arcs than this for every
                                           // 32 candidates: one step of 32 searches costs as much as six of 32 reads
constexpr int SEARCHED = -1, READ = -2;    // what happens to the row of a candidate outside the matrix
constexpr int ROW_ILP = 4;                 // arcs of those rows in flight per thread
constexpr int WARP_SIEVE = 256, CTA_SIEVE = 1024;  // words of the candidate filter
constexpr int CTA_ROWS = 4;                // rows a warp of a CTA takes at a time
constexpr int CTA_P = 1216;                // candidates of a CTA's vertex with a matrix ...
constexpr int CTA_P3 = 24576;              // ... and without (triangles)
constexpr int WARP_TEAM = 256, CTA_TEAM = 512, CTA_TEAM3 = 1024;  // threads (CTA_TEAM3: triangles)
constexpr size_t CTA_LISTS = 2 * 4 * CTA_P + 4 * (size_t)CTA_P * (CTA_P / 32 + 1);
constexpr size_t CTA_SMEM = CTA_LISTS + 4 * CTA_SIEVE;
static_assert((CTA_P / 32 + 1) % 2 == 1 && WARP_STRIDE % 2 == 1, "an odd row stride spreads rows over the banks");
static_assert(2 * 4 * (size_t)CTA_P3 <= CTA_LISTS, "triangles' candidates fit the same shared memory");

struct TdsCtl {
    long long round, size, best_round, best_size, n_min_rule;
    long long f, bf;           // clique counts
    long long gpo_le, gpo_lt;  // tau_max's integer forms (Algorithm 3)
    long long T;               // this round removes live w <= T
    long long kind;            // 0 main round, 1 minimum rule, 2 trim round
    long long minw;            // minimum live weight before the round
    long long ucnt;            // |U_i|
    long long df;              // cliques that die in the round
    int status;                // 0 running, 1 done
    int error;
    int nbig;                  // vertices left to the CTA launch
    int blocks;                // blocks of the closing launch that are through
    int core_thr, ncore;       // the adjacency matrix takes degrees >= core_thr
};

struct TdsArgs {
    long long n;
    const long long *rp;
    const int *col;
    const int *hubs;
    long long *w;
    int *pr;
    int *front;
    int *big;        // vertices left to the CTA launch
    int *ci;         // row of the adjacency matrix, -1: none
    unsigned *bits;  // [CORE_MAX][CORE_WORDS]
    int *hist;       // [DEG_BINS]
    TdsCtl *ctl;
    long long *tr_f, *tr_size, *tr_peeled;
    long long tr_cap;
    long long kD, D;
    int gpo, lpo;
    int q;  // clique size (3 for TDS)
    long long max_rounds;
};

__device__ __forceinline__ int head(const TdsArgs &A, long long p) { return arc_head(A.col[p], A.hubs); }

// first position in v's row whose neighbour id exceeds x
__device__ __forceinline__ long long row_after(const TdsArgs &A, int v, int x) {
    long long lo = A.rp[v], hi = A.rp[v + 1];
    while (lo < hi) {
        const long long mid = lo + ((hi - lo) >> 1);
        if (head(A, mid) <= x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ bool in_row(const TdsArgs &A, int v, int x) {
    const long long p = row_after(A, v, x - 1);
    return p < A.rp[v + 1] && head(A, p) == x;
}

// are x and y adjacent?  cx, cy: their rows of the adjacency matrix, or -1
__device__ __forceinline__ bool adjacent(const TdsArgs &A, int x, int cx, int y, int cy) {
    if (cx >= 0 && cy >= 0) return (A.bits[cx * CORE_WORDS + (cy >> 5)] >> (cy & 31)) & 1u;
    return cx < 0 ? in_row(A, x, y) : in_row(A, y, x);
}

// ------------------------------------------------------------------ set-up

__global__ void k_tds_reset(TdsArgs A) {
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, dt = (long long)gridDim.x * blockDim.x;
    for (long long u = t0; u < A.n; u += dt) {
        A.w[u] = 0;
        A.pr[u] = DUPIN_LIVE;
    }
    for (long long x = t0; x < DEG_BINS; x += dt) A.hist[x] = 0;
    if (t0 == 0) {
        TdsCtl z;
        memset(&z, 0, sizeof(z));
        z.gpo_lt = -1;
        z.size = A.n;
        z.minw = 0x7fffffffffffffffLL;
        *A.ctl = z;
    }
}

__global__ void k_core_hist(TdsArgs A) {
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < A.n; u += (long long)gridDim.x * blockDim.x) {
        const long long d = A.rp[u + 1] - A.rp[u];
        atomicAdd(&A.hist[d < DEG_BINS - 1 ? (int)d : DEG_BINS - 1], 1);
    }
}

// the lowest degree at which no more than CORE_MAX vertices lie (one block of
// 1024: four bins per thread, a scan from the top)
__global__ void __launch_bounds__(1024) k_core_threshold(TdsArgs A) {
    __shared__ long long s_w[32];
    __shared__ int s_best;
    const int t = threadIdx.x;
    if (t == 0) s_best = 0x7fffffff;
    const int b0 = DEG_BINS - 4 * (t + 1);  // this thread's bins b0 .. b0 + 3
    long long c[4], sum = 0;
    for (int k = 3; k >= 0; k--) {
        c[k] = A.hist[b0 + k];
        sum += c[k];
    }
    long long incl = warp_incl_scan64(sum);
    if ((t & 31) == 31) s_w[t >> 5] = incl;
    __syncthreads();
    long long above = incl - sum;
    for (int k = 0; k < (t >> 5); k++) above += s_w[k];
    for (int k = 3; k >= 0; k--) {
        above += c[k];
        if (above > CORE_MAX) break;
        atomicMin(&s_best, b0 + k);
    }
    __syncthreads();
    if (t == 0) A.ctl->core_thr = s_best;
}

__global__ void k_core_rows(TdsArgs A) {
    const int thr = A.ctl->core_thr;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < A.n; u += (long long)gridDim.x * blockDim.x) {
        const long long d = A.rp[u + 1] - A.rp[u];
        A.ci[u] = d >= thr ? atomicAdd(&A.ctl->ncore, 1) : -1;
    }
}

// a warp per core vertex clears its row and sets its neighbours' bits
__global__ void k_core_bits(TdsArgs A) {
    const int lane = threadIdx.x & 31;
    const long long W = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long u = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); u < A.n; u += W) {
        const int cu = A.ci[u];
        if (cu < 0) continue;
        unsigned *row = A.bits + (size_t)cu * CORE_WORDS;
        for (int k = lane; k < CORE_WORDS; k += 32) row[k] = 0;
        __syncwarp();
        for (long long p = A.rp[u] + lane; p < A.rp[u + 1]; p += 32) {
            const int cv = A.ci[head(A, p)];
            if (cv >= 0) atomicOr(&row[cv >> 5], 1u << (cv & 31));
        }
    }
}

__global__ void k_tds_start(TdsArgs A) {
    TdsCtl *c = A.ctl;
    c->round = 0;
    c->size = A.n;
    c->best_round = 0;
    c->best_size = A.n;
    c->bf = c->f;
    c->status = A.n == 0 ? 1 : 0;
    c->nbig = 0;
    if (A.tr_cap > 0) {
        A.tr_f[0] = c->f;
        A.tr_size[0] = A.n;
        A.tr_peeled[0] = 0;
    }
}

// ------------------------------------------------------------------ listing

// Which neighbours of u are candidates.  ROUND 0: the initial counts; else the
// round whose removals are expanded.
struct Keep {
    int u, r;  // r < 0: the initial counts
    long long du;
    __device__ __forceinline__ Keep(const TdsArgs &A, int u_, int r_) : u(u_), r(r_), du(A.rp[u_ + 1] - A.rp[u_]) {}
    __device__ __forceinline__ bool outranks(const TdsArgs &A, int x) const {
        const long long dx = A.rp[x + 1] - A.rp[x];
        return dx > du || (dx == du && x > u);
    }
    __device__ __forceinline__ bool operator()(const TdsArgs &A, int x) const {
        if (r < 0) return outranks(A, x);
        const int px = A.pr[x];
        if (px != r) return px > r;  // left in an earlier round, or survives this one
        return outranks(A, x);
    }
};

// v's share of u's cliques: t of them hold v
__device__ __forceinline__ void credit(const TdsArgs &A, int v, unsigned long long t, int r) {
    if (t == 0) return;
    if (r < 0) atomicAdd((unsigned long long *)&A.w[v], t);
    else if (A.pr[v] > r) atomicAdd((unsigned long long *)&A.w[v], 0ull - t);
}

// The M-cliques y_0 < y_1 < ... < y_{M-1} that lie in the rows row[0..D] (D
// chosen members besides the first row's), from word 'w0' on and above the
// bits that 'first' leaves in it.
template <int D, int M>
__device__ __forceinline__ unsigned long long cliques_in(const unsigned *rows, int stride, int words,
                                                         const unsigned *(&row)[M], int w0, unsigned first) {
    unsigned long long t = 0;
    for (int w = w0; w < words; w++) {
        unsigned b = row[0][w];
#pragma unroll
        for (int k = 1; k <= D; k++) b &= row[k][w];
        if (w == w0) b &= first;
        if (D == M - 1) {
            t += __popc(b);
        } else {
            while (b) {
                const int j = __ffs(b) - 1;
                b &= b - 1;
                row[D + 1 < M ? D + 1 : 0] = rows + (size_t)(32 * w + j) * stride;
                t += cliques_in<(D + 1 < M ? D + 1 : D), M>(rows, stride, words, row, w, j == 31 ? 0u : ~0u << (j + 1));
            }
        }
    }
    return t;
}

// the M-cliques among the neighbours of row 'v' whose first member's word is in
// [w0, w1) (M >= 2)
template <int M>
__device__ __forceinline__ unsigned long long cliques_of(const unsigned *rows, int stride, int words, int v, int w0, int w1) {
    const unsigned *row[M];
    row[0] = rows + (size_t)v * stride;
    unsigned long long t = 0;
    for (int w = w0; w < w1; w++) {
        unsigned b = row[0][w];
        while (b) {
            const int j = __ffs(b) - 1;
            b &= b - 1;
            row[1] = rows + (size_t)(32 * w + j) * stride;
            t += cliques_in<1, M>(rows, stride, words, row, w, j == 31 ? 0u : ~0u << (j + 1));
        }
    }
    return t;
}

__device__ __forceinline__ unsigned long long cliques_of(int M, const unsigned *rows, int stride, int words, int v, int w0,
                                                         int w1) {
    switch (M) {
        case 2: return cliques_of<2>(rows, stride, words, v, w0, w1);
        case 3: return cliques_of<3>(rows, stride, words, v, w0, w1);
        case 4: return cliques_of<4>(rows, stride, words, v, w0, w1);
        case 5: return cliques_of<5>(rows, stride, words, v, w0, w1);
        default: return cliques_of<6>(rows, stride, words, v, w0, w1);
    }
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long x) {
    return (unsigned long long)__shfl_sync(0xffffffffu, warp_sum64((long long)x), 0);
}

// Pairs of candidates are found in two ways.  Between two members of the adjacency
// matrix a bit tells, and a long row is searched for the other's id; but a row
// outside the matrix that is short against the number of candidates is read, and each
// neighbour looked up among the candidates: in a filter by its id's low bits,
// then by a search of their ids (increasing, as the row they come from).
// (TDS, k = 3.  Searches alone took 54 ms on a uniform graph of 300,000 vertices and
// degree 120, 18.7 ms on 1,000,000 of degree 32 and 146 ms on 50,000 of degree 400, where
// merging rows had taken 15.6, 7.2 and 28; with the reads it is 15.1, 5.4 and 34.)

// of each candidate outside the matrix: is its row read?  (returns whether this
// thread found such a one)
__device__ __forceinline__ bool pick_rows(const TdsArgs &A, const int *ids, int *cis, int p, int t, int nt) {
    const long long most = (long long)READ_ARCS * ((p + 31) >> 5);
    bool any = false;
    for (int v = t; v < p; v += nt) {
        if (cis[v] >= 0) continue;
        const bool read = A.rp[ids[v] + 1] - A.rp[ids[v]] <= most;
        cis[v] = read ? READ : SEARCHED;
        any = any || read;
    }
    return any;
}

__device__ __forceinline__ unsigned sieve_bit(int x) { return 1u << (x & 31); }
template <int WORDS>
__device__ __forceinline__ int sieve_word(int x) { return (x >> 5) & (WORDS - 1); }

// One warp: the rows to be read among candidates g0 .. g0 + per - 1 (per <= 32), their
// arcs spread over the lanes; hit(v, j) for each neighbour of candidate v that is
// candidate j.
template <int WORDS, class Hit>
__device__ __forceinline__ void read_rows(const TdsArgs &A, const int *ids, const int *cis, int p, const unsigned *sieve,
                                          int g0, int per, Hit hit) {
    const int lane = threadIdx.x & 31;
    const int v = g0 + lane;
    const bool mine = lane < per && v < p && cis[v] == READ;
    const long long start = mine ? A.rp[ids[v]] : 0;
    const int deg = mine ? (int)(A.rp[ids[v] + 1] - start) : 0;
    int before = deg;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, before, d);
        if (lane >= d) before += o;
    }
    const int all = __shfl_sync(0xffffffffu, before, 31);
    before -= deg;
    for (int k0 = lane; k0 - lane < all; k0 += 32 * ROW_ILP) {
        int t[ROW_ILP], y[ROW_ILP];
#pragma unroll
        for (int z = 0; z < ROW_ILP; z++) {
            const int k = k0 + 32 * z;
            t[z] = 0;  // the row of arc k: the last that starts at or before it
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, before, t[z] + step) <= k) t[z] += step;
            const long long at = __shfl_sync(0xffffffffu, start, t[z]) + (k - __shfl_sync(0xffffffffu, before, t[z]));
            y[z] = k < all ? A.col[at] : 0;
        }
#pragma unroll
        for (int z = 0; z < ROW_ILP; z++) {
            if (k0 + 32 * z >= all) continue;
            if (y[z] < 0) y[z] = A.hubs[-y[z] - 1];
            if (!(sieve[sieve_word<WORDS>(y[z])] & sieve_bit(y[z]))) continue;
            int lo = 0, hi = p - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (ids[mid] <= y[z]) lo = mid;
                else hi = mid - 1;
            }
            if (ids[lo] == y[z]) hit(g0 + t[z], lo);
        }
    }
}

// u's cliques by one warp; false when it has more than WARP_P candidates or too
// long a row.  Adds the sum over v of the cliques through v, (q-1) times u's, to 'sum'.
template <bool TRIANGLES, bool READS>
__device__ __forceinline__ bool warp_vertex(const TdsArgs &A, int u, int r, int *ids, int *cis, unsigned *rows,
                                            unsigned *sieve, unsigned long long &sum) {
    const int lane = threadIdx.x & 31;
    const Keep keep(A, u, r);
    const long long b = A.rp[u], e = A.rp[u + 1];
    if (e - b > LONG_ROW) return false;
    int p = 0;
    for (long long j0 = b; j0 < e; j0 += 32) {
        const long long j = j0 + lane;
        const int x = j < e ? head(A, j) : 0;
        const bool k = j < e && keep(A, x);
        const unsigned bal = __ballot_sync(0xffffffffu, k);
        if (p + __popc(bal) > WARP_P) return false;
        if (k) {
            const int at = p + __popc(bal & ((1u << lane) - 1u));
            ids[at] = x;
            cis[at] = A.ci[x];
        }
        p += __popc(bal);
    }
    const int q = TRIANGLES ? 3 : A.q;
    if (p < q - 1) return true;
    __syncwarp();
    const bool reads = READS && __any_sync(0xffffffffu, pick_rows(A, ids, cis, p, lane, 32));
    const int words = (p + 31) >> 5;
    const int stride = TRIANGLES ? 1 : WARP_STRIDE;  // triangles: a count per candidate in place of its matrix row
    if (reads) {
        for (int k = lane; k < WARP_SIEVE; k += 32) sieve[k] = 0;
        for (int k = lane; k < p * stride; k += 32) rows[k] = 0;
        __syncwarp();
        for (int v = lane; v < p; v += 32) atomicOr(&sieve[sieve_word<WARP_SIEVE>(ids[v])], sieve_bit(ids[v]));
    }
    __syncwarp();
    // pairs of candidates whose rows are not read
    for (int g0 = 0; g0 < p; g0 += 32) {
        unsigned left = __ballot_sync(0xffffffffu, g0 + lane < p && !(READS && cis[g0 + lane] == READ));
        while (left) {
            const int v = g0 + __ffs(left) - 1;
            left &= left - 1;
            const int x = ids[v], cx = cis[v];
            int t = 0;
            for (int w = 0; w < words; w++) {
                const int y = 32 * w + lane;
                const bool in = y < p && y != v && !(READS && cis[y] == READ) && adjacent(A, x, cx, ids[y], cis[y]);
                const unsigned bal = __ballot_sync(0xffffffffu, in);
                if (TRIANGLES) t += __popc(bal);
                else if (lane == 0) rows[v * stride + w] = bal;
            }
            if (TRIANGLES && lane == 0) rows[v] = t;
        }
    }
    __syncwarp();
    for (int g0 = 0; reads && g0 < p; g0 += 32)
        read_rows<WARP_SIEVE>(A, ids, cis, p, sieve, g0, 32, [&](int v, int j) {
            const bool both = cis[j] != READ;  // j's row will not tell
            if (TRIANGLES) {
                atomicAdd(&rows[v], 1u);
                if (both) atomicAdd(&rows[j], 1u);
            } else {
                atomicOr(&rows[v * stride + (j >> 5)], 1u << (j & 31));
                if (both) atomicOr(&rows[j * stride + (v >> 5)], 1u << (v & 31));
            }
        });
    __syncwarp();
    unsigned long long found = 0;
    for (int v = lane; v < p; v += 32) {
        const unsigned long long t = TRIANGLES ? rows[v] : cliques_of(q - 2, rows, stride, words, v, 0, words);
        credit(A, ids[v], t, r);
        found += t;
    }
    sum += found;
    __syncwarp();
    return true;
}

// Cliques of every vertex (r < 0) or of the round's removed vertices, a warp
// each; vertices with too many candidates are listed for the CTA launch.
__device__ __forceinline__ void add_cliques(const TdsArgs &A, unsigned long long sum, int r) {
    sum = warp_sum_u64(sum);
    if ((threadIdx.x & 31) == 0 && sum) {
        // every clique was counted once through each of its q - 1 members besides u
        const unsigned long long k = sum / (unsigned long long)(A.q - 1);
        atomicAdd((unsigned long long *)(r < 0 ? &A.ctl->f : &A.ctl->df), k);
        // u's own weight matters in the initial counts only (it leaves in a round)
    }
}

template <bool ROUND, bool TRIANGLES, bool READS>
__global__ void __launch_bounds__(WARP_TEAM, TRIANGLES ? 5 : 3) k_clq_warp(TdsArgs A) {
    __shared__ int s_ids[WARP_TEAM / 32][WARP_P], s_cis[WARP_TEAM / 32][WARP_P];
    __shared__ unsigned s_rows[WARP_TEAM / 32][TRIANGLES ? WARP_P : WARP_P * WARP_STRIDE];
    __shared__ unsigned s_sieve[READS ? WARP_TEAM / 32 : 1][WARP_SIEVE];
    const TdsCtl *c = A.ctl;
    if (ROUND && (c->status || c->error)) return;
    const int r = ROUND ? (int)(c->round + 1) : -1;
    const long long U = ROUND ? c->ucnt : A.n;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long W = (long long)gridDim.x * (WARP_TEAM / 32);
    unsigned long long total = 0;
    for (long long k = blockIdx.x * (long long)(WARP_TEAM / 32) + wid; k < U; k += W) {
        const int u = ROUND ? A.front[k] : (int)k;
        unsigned long long sum = 0;
        if (!warp_vertex<TRIANGLES, READS>(A, u, r, s_ids[wid], s_cis[wid], s_rows[wid], s_sieve[READS ? wid : 0], sum)) {
            if (lane == 0) A.big[atomicAdd(&A.ctl->nbig, 1)] = u;
            __syncwarp();
            continue;
        }
        sum = warp_sum_u64(sum);
        if (!ROUND && lane == 0 && sum) atomicAdd((unsigned long long *)&A.w[u], sum / (unsigned long long)(A.q - 1));
        if (lane == 0) total += sum;
    }
    add_cliques(A, total, r);
}

// positions of depth d (2 <= d <= QMAX - 1) start at pos_base(d): d of them,
// one in the row of each member chosen before depth d
__host__ __device__ constexpr int pos_base(int d) { return d * (d - 1) / 2 - 1; }

// first position in [p, end) whose id is at least x (end if none): doubling
// steps from p, then a binary search in the last step, so a long row is
// crossed in O(log gap) reads
__device__ __forceinline__ long long seek(const TdsArgs &A, long long p, long long end, int x) {
    if (p >= end || head(A, p) >= x) return p;
    long long lo = p, hi, step = 1;  // head(lo) < x
    for (;;) {
        hi = lo + step;
        if (hi >= end) {
            hi = end;
            break;
        }
        if (head(A, hi) >= x) break;
        lo = hi;
        step <<= 1;
    }
    lo++;  // the answer is in [lo, hi]
    while (lo < hi) {
        const long long mid = lo + ((hi - lo) >> 1);
        if (head(A, mid) < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The q-cliques {u, v, y_2, ..., y_{q-1}} with v < y_2 < ... < y_{q-1}, all in
// u's row, whose members pass 'keep' (v is the caller's: u's arc at position
// j).  c[0] = u, c[1] = v; at depth d the candidates y_d are the ids above
// c[d-1] present in the rows of c[0..d-1].  They are found by a leapfrog
// join: the rows take turns, each seeking its position to the largest id
// seen so far, until d rows in a row show the same id (rows are sorted, so
// every position only moves forward and the largest id only grows; a long
// row is crossed by doubling steps).  'emit' gets the q members in c[0..q-1].
template <class Keep, class Emit>
__device__ void clique_walk(const TdsArgs &A, int q, int u, long long j, long long e, int v, Keep keep, Emit emit) {
    int c[QMAX];
    long long end[QMAX];
    long long pos[pos_base(QMAX)];
    c[0] = u;
    c[1] = v;
    end[0] = e;
    end[1] = A.rp[v + 1];
    pos[pos_base(2)] = j + 1;
    pos[pos_base(2) + 1] = row_after(A, v, v);
    int d = 2;
    while (d >= 2) {
        long long *P = pos + pos_base(d);
        bool found = false;
        int y = 0;
        if (P[0] < end[0]) {
            y = head(A, P[0]);
            int agree = 1, t = 1;  // rows in turn that show y
            for (;;) {
                if (agree == d) {  // y is in every row
                    if (keep(y)) {
                        found = true;
                        break;
                    }
                    if (++P[0] >= end[0]) break;
                    y = head(A, P[0]);
                    agree = 1;
                    t = 1;
                    continue;
                }
                P[t] = seek(A, P[t], end[t], y);
                if (P[t] >= end[t]) break;  // a row is used up: no candidate left at this depth
                const int h = head(A, P[t]);
                if (h == y) {
                    agree++;
                } else {
                    y = h;
                    agree = 1;
                }
                t = t + 1 == d ? 0 : t + 1;
            }
        }
        if (!found) {
            d--;
            continue;
        }
        P[0]++;  // this depth resumes after y
        c[d] = y;
        if (d == q - 1) {
            emit(c);
            continue;
        }
        long long *N = pos + pos_base(d + 1);
        for (int t = 0; t < d; t++) N[t] = P[t];
        N[d] = row_after(A, y, y);
        end[d] = A.rp[y + 1];
        d++;
    }
}


// Vertices with more candidates than a warp takes, a CTA each.
template <bool ROUND, bool TRIANGLES, bool READS>
__global__ void __launch_bounds__(TRIANGLES ? CTA_TEAM3 : CTA_TEAM, 1) k_clq_cta(TdsArgs A) {
    extern __shared__ int s_mem[];
    constexpr int TEAM = TRIANGLES ? CTA_TEAM3 : CTA_TEAM;
    constexpr int NW = TEAM / 32;
    __shared__ int s_cnt[NW];
    __shared__ unsigned long long s_sum;
    const TdsCtl *c = A.ctl;
    if (ROUND && (c->status || c->error)) return;
    const int r = ROUND ? (int)(c->round + 1) : -1;
    const int nbig = c->nbig;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int q = TRIANGLES ? 3 : A.q;
    const int cap = TRIANGLES ? CTA_P3 : CTA_P;
    int *ids = s_mem, *cis = s_mem + cap;
    unsigned *rows = (unsigned *)(cis + cap), *sieve = (unsigned *)s_mem + CTA_LISTS / 4;
    unsigned long long total = 0;
    for (int k = blockIdx.x; k < nbig; k += gridDim.x) {
        const int u = A.big[k];
        const Keep keep(A, u, r);
        const long long b = A.rp[u], e = A.rp[u + 1];
        __syncthreads();
        if (tid == 0) s_sum = 0;
        int p = 0;
        for (long long j0 = b; j0 < e && p <= cap; j0 += TEAM) {  // candidates in id order
            const long long j = j0 + tid;
            const int x = j < e ? head(A, j) : 0;
            const bool kp = j < e && keep(A, x);
            const unsigned bal = __ballot_sync(0xffffffffu, kp);
            __syncthreads();
            if (lane == 0) s_cnt[wid] = __popc(bal);
            __syncthreads();
            int at = p, all = 0;
            for (int o = 0; o < NW; o++) {
                if (o < wid) at += s_cnt[o];
                all += s_cnt[o];
            }
            at += __popc(bal & ((1u << lane) - 1u));
            if (kp && at < cap) {
                ids[at] = x;
                cis[at] = A.ci[x];
            }
            p += all;
        }
        __syncthreads();
        unsigned long long mine = 0;  // this thread's part of the cliques through each candidate
        if (p > cap) {  // too many candidates for shared memory: walk the rows
            for (long long j = b + tid; j < e; j += TEAM) {
                const int v = head(A, j);
                if (!keep(A, v)) continue;
                clique_walk(A, q, u, j, e, v, [&](int x) { return keep(A, x); }, [&](const int *m) {
                    mine += q - 1;
                    for (int t = 1; t < q; t++) credit(A, m[t], 1, r);
                });
            }
        } else if (p >= q - 1) {
            const int words = (p + 31) >> 5, stride = words | 1;
            const bool reads = READS && __syncthreads_or(pick_rows(A, ids, cis, p, tid, TEAM));
            if (reads) {
                for (int w = tid; w < CTA_SIEVE; w += TEAM) sieve[w] = 0;
                if (!TRIANGLES)
                    for (int w = tid; w < p * stride; w += TEAM) rows[w] = 0;
                __syncthreads();
                for (int v = tid; v < p; v += TEAM) atomicOr(&sieve[sieve_word<CTA_SIEVE>(ids[v])], sieve_bit(ids[v]));
            }
            for (int v = wid; v < p; v += NW) {
                const int x = ids[v], cx = cis[v];
                if (READS && cx == READ) continue;
                int t = 0;
                for (int w = 0; w < words; w++) {
                    const int y = 32 * w + lane;
                    const unsigned bal = __ballot_sync(
                        0xffffffffu, y < p && y != v && !(READS && cis[y] == READ) && adjacent(A, x, cx, ids[y], cis[y]));
                    if (TRIANGLES) t += __popc(bal);
                    else if (lane == 0) rows[(size_t)v * stride + w] = bal;
                }
                if (TRIANGLES && lane == 0) {
                    credit(A, x, (unsigned long long)t, r);
                    mine += (unsigned long long)t;
                }
            }
            __syncthreads();
            for (int g0 = CTA_ROWS * wid; reads && g0 < p; g0 += CTA_ROWS * NW)
                read_rows<CTA_SIEVE>(A, ids, cis, p, sieve, g0, CTA_ROWS, [&](int v, int j) {
                    const bool both = cis[j] != READ;  // j's row will not tell
                    if (TRIANGLES) {
                        credit(A, ids[v], 1, r);
                        if (both) credit(A, ids[j], 1, r);
                        mine += both ? 2 : 1;
                    } else {
                        atomicOr(&rows[(size_t)v * stride + (j >> 5)], 1u << (j & 31));
                        if (both) atomicOr(&rows[(size_t)j * stride + (v >> 5)], 1u << (v & 31));
                    }
                });
            if (reads) __syncthreads();
            if (!TRIANGLES) {
                for (int v = wid; v < p; v += NW) {  // lanes share the first member's words
                    unsigned long long t = 0;
                    for (int w = lane; w < words; w += 32) t += cliques_of(q - 2, rows, stride, words, v, w, w + 1);
                    t = warp_sum_u64(t);
                    if (lane == 0) {
                        credit(A, ids[v], t, r);
                        mine += t;
                    }
                }
            }
        }
        mine = warp_sum_u64(mine);
        if (lane == 0 && mine) atomicAdd(&s_sum, mine);
        __syncthreads();
        if (tid == 0) {
            if (!ROUND && s_sum) atomicAdd((unsigned long long *)&A.w[u], s_sum / (unsigned long long)(q - 1));
            total += s_sum;
        }
    }
    if (wid == 0) add_cliques(A, total, r);
}

// ------------------------------------------------------------------ rounds

__device__ __forceinline__ long long tds_floor(u128 x, u128 y) {
    const u128 q = x / y;
    return q > (u128)0x7fffffffffffffffULL ? 0x7fffffffffffffffLL : (long long)q;
}

// ceil(x / y) - 1 (the largest integer strictly below x / y), -1 for x = 0
__device__ __forceinline__ long long tds_below(u128 x, u128 y) {
    if (x == 0) return -1;
    return tds_floor(x - 1, y);
}

// f, |S|, the trace and the best prefix of the round just expanded
__device__ void close_round(const TdsArgs &A) {
    TdsCtl *c = A.ctl;
    if (c->ucnt == 0) {  // cannot happen (Lemma 4.2 / minimum rule)
        c->error = DUPIN_ERR_NO_PROGRESS;
        return;
    }
    const long long i = c->round + 1;
    c->f -= c->df;
    c->size -= c->ucnt;
    c->round = i;
    c->n_min_rule += c->kind == 1 ? 1 : 0;
    if (c->size > 0 &&
        (u128)(unsigned long long)c->f * (unsigned long long)c->best_size >
            (u128)(unsigned long long)c->bf * (unsigned long long)c->size) {
        c->bf = c->f;
        c->best_size = c->size;
        c->best_round = i;
    }
    if (i < A.tr_cap) {
        A.tr_f[i] = c->f;
        A.tr_size[i] = c->size;
        A.tr_peeled[i] = c->ucnt;
    }
    if (c->size == 0) c->status = 1;
}

__device__ void plan_round(const TdsArgs &A) {
    TdsCtl *c = A.ctl;
    if (c->round + 1 > A.max_rounds) {
        c->error = DUPIN_ERR_NO_PROGRESS;
        return;
    }
    const u128 f = (u128)(unsigned long long)c->f, size = (u128)(unsigned long long)c->size;
    const long long m = c->minw;
    const long long below_g = tds_below(f, size);
    if (A.lpo && c->round > 0 && m <= below_g) {  // Algorithm 4: some live w < g(S)
        c->T = below_g > c->gpo_lt ? below_g : c->gpo_lt;
        c->kind = 2;
    } else {
        long long T = tds_floor((u128)(unsigned long long)A.kD * f, (u128)(unsigned long long)A.D * size);
        if (A.gpo) {  // Algorithm 3: tau_max refined at every main round
            const u128 num = (u128)(unsigned long long)A.D * f, den = (u128)(unsigned long long)A.kD * size;
            const long long le = tds_floor(num, den), lt = tds_below(num, den);
            if (le > c->gpo_le) c->gpo_le = le;
            if (lt > c->gpo_lt) c->gpo_lt = lt;
            if (c->gpo_le > T) T = c->gpo_le;
        }
        c->kind = 0;
        if (m > T) {  // the threshold selects nobody: the minimum rule
            T = m;
            c->kind = 1;
        }
        c->T = T;
    }
    c->ucnt = 0;
    c->df = 0;
    c->nbig = 0;
}

// the minimum live weight; the last block through closes the round (unless
// none has run yet) and plans the next
__global__ void k_tds_close(TdsArgs A, int first) {
    TdsCtl *c = A.ctl;
    if (c->status || c->error) return;
    long long m = 0x7fffffffffffffffLL;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < A.n; u += (long long)gridDim.x * blockDim.x)
        if (A.pr[u] == DUPIN_LIVE && A.w[u] < m) m = A.w[u];
    m = warp_min64(m);
    if ((threadIdx.x & 31) == 0 && m != 0x7fffffffffffffffLL) atomicMin(&c->minw, m);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&c->blocks, 1) == (int)gridDim.x - 1) {
        __threadfence();
        c->blocks = 0;
        c->minw = atomicMin(&c->minw, 0x7fffffffffffffffLL);  // read where the other blocks wrote
        if (!first) close_round(A);
        if (!c->status && !c->error) plan_round(A);
        c->minw = 0x7fffffffffffffffLL;
    }
}

__global__ void k_tds_select(TdsArgs A) {
    const TdsCtl *c = A.ctl;
    if (c->status || c->error) return;
    const long long T = c->T;
    const int r = (int)(c->round + 1);
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long b = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); b < A.n; b += stride) {
        const long long u = b + lane;
        const bool sel = u < A.n && A.pr[u] == DUPIN_LIVE && A.w[u] <= T;
        const unsigned m = __ballot_sync(0xffffffffu, sel);
        if (!m) continue;
        long long base = 0;
        if (lane == 0) base = (long long)atomicAdd((unsigned long long *)&A.ctl->ucnt, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (sel) {
            A.pr[u] = r;
            A.front[base + __popc(m & ((1u << lane) - 1u))] = (int)u;
        }
    }
}

__global__ void k_tds_mask(const int *pr, long long n, const TdsCtl *c, uint8_t *mask) {
    const long long br = c->best_round;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x)
        mask[u] = (long long)pr[u] > br ? 1 : 0;
}

// the CTA kernels' shared memory, once per device
int set_clique_smem() {
    static std::mutex mu;
    static bool done[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return dupin_fail(DUPIN_ERR_CUDA, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(mu);
    if (done[dev]) return DUPIN_OK;
    for (const void *f : {(const void *)k_clq_cta<false, false, false>, (const void *)k_clq_cta<true, false, false>,
                          (const void *)k_clq_cta<false, true, false>, (const void *)k_clq_cta<true, true, false>,
                          (const void *)k_clq_cta<false, false, true>, (const void *)k_clq_cta<true, false, true>,
                          (const void *)k_clq_cta<false, true, true>, (const void *)k_clq_cta<true, true, true>}) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CTA_SMEM);
        if (e != cudaSuccess) return dupin_cuda_fail(e, "cudaFuncSetAttribute(k_clq_cta)");
    }
    done[dev] = true;
    return DUPIN_OK;
}

}  // namespace

// dupin_peel for the metrics DUPIN_TDS and DUPIN_KCLIDS (parameters checked by the caller).
int tds_peel(dupin_graph *g, const dupin_params *p, dupin_result *r, cudaStream_t s) {
    const long long n = g->n;
    const long long max_rounds = p->max_rounds > 0 ? p->max_rounds : n + 1;
    const long long tr_cap = std::min<long long>(max_rounds, n) + 1;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device);
    TdsArgs A;
    memset(&A, 0, sizeof(A));
    A.n = n;
    A.rp = g->rp;
    A.col = g->col;
    A.hubs = g->hubs;
    A.kD = (long long)p->k_mult * (p->eps_den + p->eps_num);
    A.D = p->eps_den;
    A.gpo = (p->flags & (DUPIN_GPO | DUPIN_LPO)) ? 1 : 0;
    A.lpo = (p->flags & DUPIN_LPO) ? 1 : 0;
    A.q = p->metric == DUPIN_KCLIDS ? p->clique_q : 3;
    A.max_rounds = max_rounds;
    A.tr_cap = tr_cap;
    int rc = set_clique_smem();
    if (rc) return rc;
    // one block from the scratch pool (the default pool would give it back to the
    // driver at every call's end)
    size_t at = 0;
    auto part = [&](size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_w = part(8 * (size_t)n), o_pr = part(4 * (size_t)n), o_front = part(4 * (size_t)n),
                 o_big = part(4 * (size_t)n), o_ci = part(4 * (size_t)n), o_ctl = part(sizeof(TdsCtl)),
                 o_trf = part(8 * (size_t)tr_cap), o_trs = part(8 * (size_t)tr_cap), o_trp = part(8 * (size_t)tr_cap),
                 o_hist = part(4 * DEG_BINS), o_mask = part((size_t)n),
                 o_bits = part(4 * (size_t)CORE_WORDS * (size_t)std::min<long long>(n, CORE_MAX));
    unsigned char *buf = nullptr;
    cudaError_t e = scratch_alloc((void **)&buf, at, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return dupin_fail(e == cudaErrorMemoryAllocation ? DUPIN_ERR_OOM : DUPIN_ERR_CUDA,
                          std::string("clique peel state: ") + cudaGetErrorString(e));
    }
    auto release = [&]() { scratch_free(buf, s); };
    A.w = (long long *)(buf + o_w);
    A.pr = (int *)(buf + o_pr);
    A.front = (int *)(buf + o_front);
    A.big = (int *)(buf + o_big);
    A.ci = (int *)(buf + o_ci);
    A.ctl = (TdsCtl *)(buf + o_ctl);
    A.tr_f = (long long *)(buf + o_trf);
    A.tr_size = (long long *)(buf + o_trs);
    A.tr_peeled = (long long *)(buf + o_trp);
    A.hist = (int *)(buf + o_hist);
    A.bits = (unsigned *)(buf + o_bits);
    // grids: as many blocks as there is work for, up to a few per SM
    const int vgrid = (int)std::max<long long>(1, std::min<long long>(sms * 8, (n + 255) / 256));
    const int cgrid = (int)std::max<long long>(1, std::min<long long>(sms, (n + 1023) / 1024));
    const int wgrid = (int)std::max<long long>(1, std::min<long long>(sms * 8, (n + WARP_TEAM / 32 - 1) / (WARP_TEAM / 32)));
    // the two listing launches, in the form for this peel: 'round', triangles or
    // not, rows read or not (up to CORE_MAX vertices all are in the matrix)
    auto list = [&](auto round, auto triangles, auto reads) {
        constexpr bool R = decltype(round)::value, T = decltype(triangles)::value, D = decltype(reads)::value;
        k_clq_warp<R, T, D><<<wgrid, WARP_TEAM, 0, s>>>(A);
        k_clq_cta<R, T, D><<<sms, T ? CTA_TEAM3 : CTA_TEAM, CTA_SMEM, s>>>(A);
    };
    auto listing = [&](auto round) {
        if (A.q == 3 && n > CORE_MAX) list(round, std::true_type{}, std::true_type{});
        else if (A.q == 3) list(round, std::true_type{}, std::false_type{});
        else if (n > CORE_MAX) list(round, std::false_type{}, std::true_type{});
        else list(round, std::false_type{}, std::false_type{});
    };
    k_tds_reset<<<vgrid, 256, 0, s>>>(A);
    k_core_hist<<<vgrid, 256, 0, s>>>(A);
    k_core_threshold<<<1, 1024, 0, s>>>(A);
    k_core_rows<<<vgrid, 256, 0, s>>>(A);
    k_core_bits<<<wgrid, WARP_TEAM, 0, s>>>(A);
    listing(std::false_type{});
    k_tds_start<<<1, 1, 0, s>>>(A);
    k_tds_close<<<cgrid, 1024, 0, s>>>(A, 1);
    TdsCtl hc;
    int group = 2;
    for (long long done_rounds = 0;; done_rounds += group, group = group < 32 ? 2 * group : 32) {
        for (int j = 0; j < group; j++) {
            k_tds_select<<<vgrid, 256, 0, s>>>(A);
            listing(std::true_type{});
            k_tds_close<<<cgrid, 1024, 0, s>>>(A, 0);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, A.ctl, sizeof(hc), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
            rc = dupin_cuda_fail(e, "clique peel rounds");
            break;
        }
        if (hc.error || hc.status) break;
        if (done_rounds > max_rounds + 64) {  // the device stops itself first; a guard only
            rc = dupin_fail(DUPIN_ERR_NO_PROGRESS, "max_rounds reached before the set became empty");
            break;
        }
    }
    if (rc == DUPIN_OK && hc.error)
        rc = dupin_fail(hc.error, hc.error == DUPIN_ERR_NO_PROGRESS ? "max_rounds reached before the set became empty"
                                                                    : "clique peel failed");
    if (rc == DUPIN_OK) {
        r->n_rounds = hc.round;
        r->best_round = hc.best_round;
        r->best_size = hc.best_size;
        r->best_f_hi = 0;
        r->best_f_lo = (unsigned long long)hc.bf;
        r->best_density = hc.best_size > 0 ? (double)hc.bf / (double)hc.best_size : 0.0;
        r->n_min_rule = hc.n_min_rule;
        r->n_bulk_rounds = 0;
        r->tail_arcs = 0;
        r->tail_ctas = 0;
        for (int j = 0; j < 4; j++) r->phase_ms[j] = 0.f;
        const bool dev = (p->flags & DUPIN_RESULT_DEVICE) != 0;
        const cudaMemcpyKind kind = dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
        if (r->best_mask && n > 0) {
            uint8_t *mk = buf + o_mask;
            k_tds_mask<<<vgrid, 256, 0, s>>>(A.pr, n, A.ctl, dev ? r->best_mask : mk);
            if (!dev) e = cudaMemcpyAsync(r->best_mask, mk, (size_t)n, cudaMemcpyDeviceToHost, s);
        }
        if (e == cudaSuccess && r->peel_round && n > 0)
            e = cudaMemcpyAsync(r->peel_round, A.pr, 4 * (size_t)n, kind, s);
        const long long nt = hc.round + 1;
        const long long cnt = std::min<long long>(nt, r->trace_cap);
        if (e == cudaSuccess && cnt > 0) {
            // f of each S_i as a (hi, lo) pair: the counts are below 2^63
            if (r->trace_f_lo) e = cudaMemcpyAsync(r->trace_f_lo, A.tr_f, 8 * (size_t)cnt, kind, s);
            if (e == cudaSuccess && r->trace_f_hi) {
                if (dev) e = cudaMemsetAsync(r->trace_f_hi, 0, 8 * (size_t)cnt, s);
                else memset(r->trace_f_hi, 0, 8 * (size_t)cnt);
            }
            if (e == cudaSuccess && r->trace_size) e = cudaMemcpyAsync(r->trace_size, A.tr_size, 8 * (size_t)cnt, kind, s);
            if (e == cudaSuccess && r->trace_peeled)
                e = cudaMemcpyAsync(r->trace_peeled, A.tr_peeled, 8 * (size_t)cnt, kind, s);
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = dupin_cuda_fail(e, "clique peel results");
        if (rc == DUPIN_OK && (r->trace_f_hi || r->trace_f_lo || r->trace_size || r->trace_peeled) &&
            r->trace_cap < nt)
            rc = dupin_fail(DUPIN_ERR_BUFFER_TOO_SMALL, "trace_cap < n_rounds + 1 (n_rounds is filled)");
    }
    release();
    return rc;
}
