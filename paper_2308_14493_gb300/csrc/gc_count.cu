// gc_count.cu -- PGD-style counting over the flagged region union graph
// (steps a3..a7): per-edge triangles, 4-cliques, 4-cycles, the per-edge and
// per-vertex terms, and the closed forms that turn them into the six induced
// graphlet counts of G_a and G_b (Sec. 3 "PGD Algorithm"; Algorithm 2).
//
// Non-induced sums per graph X (d = degree in X, t_uv = |N(u) n N(v)|):
//   P  = sum_{uv} (d_u-1)(d_v-1) - t_uv        3-paths
//   S  = sum_v C(d_v,3)                        3-stars
//   TT = 1/2 sum_{uv} t_uv (d_u+d_v-4)         tailed triangles
//   D  = sum_{uv} C(t_uv,2)                    diamonds
//   K  = #4-cliques,  Q = #4-cycles (not necessarily induced)
// Induced counts invert the containment of each graphlet in the larger ones:
//   g6 = K, g5 = D-6K, g3 = Q-g5-3K, g4 = TT-4g5-12K,
//   g2 = S-g4-2g5-4K, g1 = P-2g4-4g3-6g5-12K.
//
// Orientation: an edge points from its lower to its higher internal id.
//
// Triangles and 4-cliques, root-centred.  For a root u with out-list
// X = N+(u) (k entries), every v = X[q] is probed: each entry y of N+(v)
// that is also in X closes the triangle (u, v, y), listed exactly once
// (u < v < y).  It sets bit p = pos(y) of the local row q, and credits its
// three edges: (u,v) and (u,y) through the rows and a per-root counter, (v,y)
// by one 64-bit atomic.  The rows are the adjacency of N+(u) as bitmasks, so
// the 4-cliques through u are sum over bits p of row q of
// popcount(row_q & row_p).  Roots are binned by k: a warp (k <= 32), a block
// (k <= TRI_KM), or per-edge merging (larger k).
//
// 4-cycles, pivot-centred.  Each 4-cycle is counted once at its highest
// vertex u: for every w < u, c_w = #{v in N(u) n N(w): v < u}, and the
// pivot contributes sum_w C(c_w, 2).  Counters are incremented one wedge
// u-v-w at a time and the increment returns the old value c, so the pivot's
// sum is accumulated on the fly as sum of old values (C(c+1,2) - C(c,2) = c);
// no reduction pass is needed.  Pivots are binned by the wedge bound
// w~ = sum of the degrees of the lower neighbours: registers (w~ <= 32, equal
// endpoints grouped by __match_any_sync), a per-warp hash table in shared
// memory, and the block kernels of gc_cycles.cu beyond.
//
// An edge set counts for G_a (G_b) only if all its entries carry FLAG_A
// (FLAG_B), so one walk serves both graphs.
#include <algorithm>

#include "gc_c4.cuh"
#include "gc_internal.cuh"
#include "gc_kernels.cuh"

namespace gcx {

__global__ void k_reset_count(Ctl* c) {
    pdl_enter();
    int t = threadIdx.x;
    if (t < NACC) c->acc[t] = 0;
    for (int i = t; i < NACC * ACC_STRIPES; i += blockDim.x) (&c->accs[0][0])[i] = 0;
    if (t < NWORK) c->work[t] = 0;
    if (t < NBINS) c->nbin[t] = 0;
    for (int i = t; i < 128; i += blockDim.x) c->c4_hist[i] = c->c4_cur[i] = 0;
    if (t == 0) {
        c->maxdeg = 0;
        c->c4_wt = c->c4_wmax = 0;
        c->ts[2] = global_ns();
        close_levels(c);
        for (int i = 3; i < 10; i++)
            if (i != 7) c->ts[i] = 0;
    }
}

__global__ void k_zero_u64(unsigned long long* __restrict__ a, const long long* d_len) {
    pdl_enter();
    long long n = *d_len;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        a[i] = 0;
}

__device__ __forceinline__ unsigned long long flag_inc(uint32_t f) {
    return ((f & FLAG_A) ? (1ull << 32) : 0ull) | ((f & FLAG_B) ? 1ull : 0ull);
}

// index of id y in the sorted entries s[0..k), or -1 (the first probes of
// all lanes hit the same entries, which shared memory broadcasts)
__device__ __forceinline__ int find_pos(const uint32_t* s, int k, uint32_t y) {
    int lo = 0, hi = k;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (vid(s[mid]) < y) lo = mid + 1;
        else hi = mid;
    }
    return (lo < k && vid(s[lo]) == y) ? lo : -1;
}

// largest q in [0, k) with pre[q] <= t (pre[0] = 0 <= t < pre[k])
__device__ __forceinline__ int find_seg(const int* pre, int k, int t) {
    int lo = 0, hi = k;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (pre[mid] <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// ---- binning ---------------------------------------------------------------

// Tier of a 4-cycle pivot with wedge bound wt.
__device__ __forceinline__ int c4_bin(const Tuning& t, long long wt) {
    return wt <= t.c4_reg_max                         ? BIN_C4_REG
           : wt <= t.c4_warp_max                      ? BIN_C4_WARP
           : wt <= min(t.c4_block_max, C4B_SMALL_MAX) ? BIN_C4_BSMALL
           : wt <= t.c4_block_max                     ? BIN_C4_BLOCK
           : wt <= t.c4_cta_max                       ? BIN_C4_BIG
                                                      : BIN_C4_DENSE;
}
// Bucket of a wedge bound, two per octave, the largest bounds first.
__device__ __forceinline__ int wedge_bucket(long long w) {
    const int lg = 63 - __clzll(w | 1);
    return 127 - (2 * lg + (lg > 0 ? (int)((w >> (lg - 1)) & 1) : 0));
}

// Wedge bound of every 4-cycle pivot: w~(u) = sum of the union-graph degrees
// of its lower neighbours.  Bound by the latency of entry and degree loads.
// Up to four vertices a warp, a warp takes one at a time.  Beyond, eight lanes
// take a vertex and a warp 32, since a warp per vertex has one short row in
// flight (1.53 ms on a graph of 4.8 M vertices and 69 M edges, 0.84 now), and
// long lists wait for the whole block.  The sums over the largest tier, which
// plan its chunks, are made here, so that the plan need not wait for the bins.
constexpr int WB_LONG = 256;
constexpr int WB_LONGS = 256;  // a block's list of them (a warp takes each further one)
__global__ void __launch_bounds__(256)
    k_wedge_bound(Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                  const uint32_t* __restrict__ U_col, const int32_t* __restrict__ U_split,
                  long long* __restrict__ U_wt, Tuning t) {
    pdl_enter();
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = (gridDim.x * blockDim.x) >> 5;
    unsigned long long wsum = 0, wmax = 0;  // of the pivots for shared memory
    auto put = [&](int32_t u, int sp, long long w) {
        U_wt[u] = w;
        if (sp >= 2 && c4_bin(t, w) == BIN_C4_DENSE) {
            wsum += (unsigned long long)w;
            wmax = max(wmax, (unsigned long long)w);
            atomicAdd(&c->c4_hist[wedge_bucket(w)], 1u);
        }
    };
    auto sum = [&](long long b, int len, int first, int step) {
        long long part = 0;
#pragma unroll 4
        for (int j = first; j < len; j += step) {
            const uint32_t v = vid(U_col[b + j]);
            part += U_off[v + 1] - U_off[v];
        }
        return part;
    };
    auto by_warp = [&](int32_t u, int sp, long long rb) {
        long long w = sp >= 2 ? sum(rb, sp, lane, 32) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(FULL, w, o);
        if (lane == 0) put(u, sp, w);
    };
    __shared__ int32_t s_long[WB_LONGS];
    __shared__ int s_nlong;
    __shared__ long long s_part[8];
    if (threadIdx.x == 0) s_nlong = 0;
    __syncthreads();
    const bool few = nW <= 4 * nwarps;
    if (few)
        for (long long i = warp; i < nW; i += nwarps) {
            const int32_t u = wlist[i];
            by_warp(u, U_split[u], U_off[u]);
        }
    // eight quads of neighbouring vertices, spread over the ids
    const int quads = few ? 0 : (nW + 3) / 4;
    for (long long base = warp; base < quads; base += 8 * nwarps) {
        const long long i = 4 * (base + (lane >> 2) * nwarps) + (lane & 3);
        int32_t u = -1;
        int sp = 0;
        long long rb = 0;
        bool over = false;  // long, and the block's list is full
        if (i < nW) {
            u = wlist[i];
            sp = U_split[u];
            rb = U_off[u];
            if (sp > WB_LONG) {
                const int at = atomicAdd(&s_nlong, 1);
                over = at >= WB_LONGS;
                if (!over) s_long[at] = u;
            }
        }
#pragma unroll 2
        for (int r = 0; r < 8; r++) {
            const int src = 4 * r + (lane >> 3);
            const int32_t x = __shfl_sync(FULL, u, src);
            const int len = __shfl_sync(FULL, sp, src);
            const long long b = __shfl_sync(FULL, rb, src);
            long long w = len >= 2 && len <= WB_LONG ? sum(b, len, lane & 7, 8) : 0;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) w += __shfl_xor_sync(FULL, w, o);
            if ((lane & 7) == 0 && x >= 0 && len <= WB_LONG) put(x, len, w);
        }
        for (unsigned m = __ballot_sync(FULL, over); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            by_warp(__shfl_sync(FULL, u, src), __shfl_sync(FULL, sp, src), __shfl_sync(FULL, rb, src));
        }
    }
    __syncthreads();
    const int nlong = min(s_nlong, WB_LONGS);
    for (int k = 0; k < nlong; k++) {
        const int32_t u = s_long[k];
        const int sp = U_split[u];
        const long long w = (long long)warp_sum_u64((unsigned long long)sum(U_off[u], sp, threadIdx.x, blockDim.x));
        if (lane == 0) s_part[threadIdx.x >> 5] = w;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long all = 0;
            for (int i = 0; i < (int)(blockDim.x >> 5); i++) all += s_part[i];
            put(u, sp, all);
        }
        __syncthreads();
    }
    wsum = warp_sum_u64(wsum);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wmax = max(wmax, __shfl_xor_sync(FULL, wmax, o));
    if (lane == 0 && wsum) {
        atomicAdd(&c->c4_wt, wsum);
        atomicMax(&c->c4_wmax, wmax);
    }
}

// Work bins: triangle roots by out-degree, 4-cycle pivots by w~.
__global__ void k_bin(Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                      const int32_t* __restrict__ U_split, const long long* __restrict__ U_wt,
                      int32_t* __restrict__ bins, int n, Tuning t) {
    pdl_enter();
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long nW_r = ((long long)nW + 31) & ~31ll;
    int dmax = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nW_r; i += stride) {
        const bool valid = i < nW;
        int tb = -1, cb = -1, bk = -1;
        const int32_t u = valid ? wlist[i] : 0;
        if (valid) {
            const long long rb = U_off[u], re = U_off[u + 1];
            const int split = U_split[u];
            const int k = (int)(re - rb) - split;
            dmax = max(dmax, (int)(re - rb));
            if (k >= 2)
                tb = k <= t.tri_warp_max    ? BIN_TRI_WARP
                     : k <= t.tri_small_max ? BIN_TRI_SMALL
                     : k <= t.tri_block_max ? BIN_TRI_BLOCK
                                            : BIN_TRI_MERGE;
            if (split >= 2) {
                const long long wt = U_wt[u];
                cb = c4_bin(t, wt);
                if (cb == BIN_C4_DENSE) bk = wedge_bucket(wt);
            }
        }
#pragma unroll 1
        for (int b = 0; b < NBINS; b++) {
            bool mine = valid && (tb == b || cb == b);
            unsigned m = __ballot_sync(FULL, mine);
            if (m) {
                int leader = __ffs(m) - 1, base = 0;
                if (lane == leader) base = atomicAdd(&c->nbin[b], __popc(m));
                base = __shfl_sync(FULL, base, leader);
                if (b == BIN_C4_DENSE) {  // by falling wedge bound: behind the buckets before
                    unsigned before[4], run = 0;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const unsigned x = c->c4_hist[32 * q + lane];
                        unsigned y = x;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const unsigned z = __shfl_up_sync(FULL, y, o);
                            if (lane >= o) y += z;
                        }
                        before[q] = run + y - x;
                        run += __shfl_sync(FULL, y, 31);
                    }
                    unsigned at = 0;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const unsigned z = __shfl_sync(FULL, before[q], bk & 31);
                        if ((bk >> 5) == q) at = z;
                    }
                    if (mine) bins[(size_t)b * n + at + atomicAdd(&c->c4_cur[bk], 1u)] = u;
                } else if (mine) {
                    bins[(size_t)b * n + base + __popc(m & lanemask_lt())] = u;
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_down_sync(FULL, dmax, o));
    stage_end(c, 3);
    if (lane == 0 && dmax) atomicMax(&c->maxdeg, dmax);
}

// ---- triangles and 4-cliques -------------------------------------------------

// A root's candidates (the entries of N+(v), v in X) are about twenty times its
// triangles, so the test "is y in X" is what the kernels spend their
// instructions on.  Each candidate is first looked up in a bitmap of hashed ids
// in shared memory (one load); the few that pass are queued per warp and
// located in X by binary search 32 at a time, with every lane at work.  Four
// candidates a lane are loaded together.  Rows of X's adjacency hold the
// triangles in G_a (R); D marks those in one graph only, so G_b's rows are
// R ^ D, and while D is empty both graphs have the same 4-cliques, counted
// once.  t of (u, X[q]) is popcount(row q) plus the triangles whose third
// vertex is X[q], kept as 16/16 bits (an out-list has at most TRI_KM entries).
// (Binary search of every candidate, 64-bit shared-memory atomics, which are
// compare-and-swap loops, and rows of an even stride took 16.4 ms for all three
// sizes on the 1.6M/30M graph and 16.1 ms on the 2.4M/5M graph with out-lists
// of up to 480 entries; these take 8.7 and 5.2 ms.)
struct Cand {
    int j;       // number of the candidate (its row q and slot follow from it)
    uint32_t e;  // entry (X[q], y)
};
constexpr int TQ = 32 + 4 * 32;  // queue entries per warp: less than 32 left over, then up to 128 more

__device__ __forceinline__ uint32_t tri_hash(uint32_t id, int lg) { return (id * 0x9E3779B1u) >> (32 - lg); }

// A root's lists in shared memory (k = |X|, W words a row, rows `ws` apart).
struct Root {
    const uint32_t* X;
    const long long* nb;  // start of N+(X[q])
    const int* pre;       // candidates before row q
    const uint32_t* bloom;
    uint32_t *R, *D, *cnt;
    int k, ws, lg;
};

// Locate up to 32 queued candidates in X and record their triangles; returns
// whether one was in one graph only.
__device__ __forceinline__ bool tri_record(const Root& t, const Cand* queue, int n, unsigned long long* tpack) {
    const int lane = threadIdx.x & 31;
    bool one = false;
    if (lane < n) {
        const Cand c = queue[lane];
        const int p = find_pos(t.X, t.k, vid(c.e));
        if (p >= 0) {
            const int q = find_seg(t.pre, t.k, c.j);
            const uint32_t f = t.X[q] & t.X[p] & c.e;
            const unsigned long long iv = flag_inc(f);
            if (iv) {
                const uint32_t bit = 1u << (p & 31);
                uint32_t* r = t.R + q * t.ws + (p >> 5);
                if (f & FLAG_A) atomicOr(r, bit);
                if ((f >> 30) != 3u) {
                    atomicOr(t.D + (r - t.R), bit);
                    one = true;
                }
                atomicAdd(&t.cnt[p], ((f & FLAG_A) ? 0x10000u : 0u) | (f >> 31));
                atomicAdd(&tpack[t.nb[q] + (c.j - t.pre[q])], iv);
            }
        }
    }
    return one;
}

// The candidates [base, base + 128) of a root, from row q on (the row of
// base); n entries are queued already.
__device__ __forceinline__ bool tri_chunk(const Root& t, const uint32_t* __restrict__ U_col, int base, int total, int q,
                                          Cand* queue, int& n, unsigned long long* tpack) {
    const int lane = threadIdx.x & 31;
    uint32_t e[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int j = base + 32 * i + lane;
        e[i] = 0xFFFFFFFFu;
        if (j < total) {
            while (q + 1 < t.k && t.pre[q + 1] <= j) q++;
            e[i] = U_col[t.nb[q] + (j - t.pre[q])];
        }
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const uint32_t h = tri_hash(vid(e[i]), t.lg);
        const bool pass = base + 32 * i + lane < total && ((t.bloom[h >> 5] >> (h & 31)) & 1u);
        const unsigned m = __ballot_sync(FULL, pass);
        if (pass) queue[n + __popc(m & lanemask_lt())] = Cand{base + 32 * i + lane, e[i]};
        n += __popc(m);
    }
    __syncwarp();
    bool one = false;
    while (n >= 32) {
        n -= 32;
        one |= tri_record(t, queue + n, 32, tpack);
    }
    __syncwarp();
    return one;
}

constexpr int TW = 8;  // warps per block of the warp-per-root kernel
struct WarpTri {
    long long nb[32];
    Cand queue[TQ];
    uint32_t X[32], R[32], D[32], cnt[32], bloom[32];
    int pre[33];
};

__global__ void __launch_bounds__(TW * 32) k_tri_warp(Ctl* c, const int32_t* __restrict__ list,
                                                     const long long* __restrict__ U_off,
                                                     const uint32_t* __restrict__ U_col,
                                                     const int32_t* __restrict__ U_split,
                                                     unsigned long long* __restrict__ tpack) {
    pdl_enter();
    __shared__ __align__(16) WarpTri s_w[TW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    WarpTri& S = s_w[w];
    const int cnt = c->nbin[BIN_TRI_WARP];
    unsigned long long ka = 0, kb = 0;
    for (int i = blockIdx.x * TW + w; i < cnt; i += gridDim.x * TW) {
        const int32_t u = list[i];
        const long long rb = U_off[u] + U_split[u];
        const int k = (int)(U_off[u + 1] - rb);
        const uint32_t x = lane < k ? U_col[rb + lane] : 0u;
        const uint32_t xmax = vid(__shfl_sync(FULL, x, k - 1));
        int cq = 0;
        long long nb = 0;
        if (lane < k) {
            const uint32_t v = vid(x);
            nb = U_off[v] + U_split[v];
            cq = (int)lower_bound_id(U_col + nb, U_off[v + 1] - nb, xmax + 1);
        }
        int inc = cq;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += y;
        }
        const int total = __shfl_sync(FULL, inc, 31);
        S.X[lane] = x;
        S.nb[lane] = nb;
        S.pre[lane + 1] = inc;
        if (lane == 0) S.pre[0] = 0;
        S.R[lane] = 0;
        S.D[lane] = 0;
        S.cnt[lane] = 0;
        S.bloom[lane] = 0;
        __syncwarp();
        if (lane < k) {
            const uint32_t h = tri_hash(vid(x), 10);
            atomicOr(&S.bloom[h >> 5], 1u << (h & 31));
        }
        __syncwarp();
        const Root t{S.X, S.nb, S.pre, S.bloom, S.R, S.D, S.cnt, k, 1, 10};
        int n = 0, q = 0;
        bool one = false;
        for (int base = 0; base < total; base += 128) {
            while (q + 1 < k && S.pre[q + 1] <= base) q++;
            one |= tri_chunk(t, U_col, base, total, q, S.queue, n, tpack);
        }
        one |= tri_record(t, S.queue, n, tpack);
        one = __any_sync(FULL, one);
        if (lane < k) {
            const uint32_t ra = S.R[lane];
            unsigned na = 0;
            for (uint32_t m = ra; m; m &= m - 1) na += __popc(ra & S.R[__ffs(m) - 1]);
            ka += na;
            const uint32_t rbm = ra ^ S.D[lane];
            if (one) {
                na = 0;
                for (uint32_t m = rbm; m; m &= m - 1) {
                    const int p = __ffs(m) - 1;
                    na += __popc(rbm & (S.R[p] ^ S.D[p]));
                }
            }
            kb += na;
            const uint32_t cn = S.cnt[lane];
            const unsigned long long tq =
                ((unsigned long long)(__popc(ra) + (cn >> 16)) << 32) | (__popc(rbm) + (cn & 0xFFFFu));
            if (tq) atomicAdd(&tpack[rb + lane], tq);
        }
        __syncwarp();
    }
    acc_add(c, 4, ka);
    acc_add(c, 10, kb);
    stage_end(c, 4);
}

// Shared memory of the block kernel for out-lists of up to KM entries; rows
// have an odd number of words, so that lanes on consecutive rows meet
// different banks.
template <int KM, int THREADS>
struct BlockTri {
    static constexpr int LG = KM <= 128 ? 12 : 14;  // bitmap bits: at most 3 % of them set
    long long nb[KM];
    Cand queue[THREADS / 32][TQ];
    uint32_t X[KM], cnt[KM], bloom[1 << (LG - 5)];
    int pre[KM + 1];
    uint32_t R[KM * (KM / 32 + 1)], D[KM * (KM / 32 + 1)];
};

constexpr int TRI_SMALL_THREADS = 256, TRI_BIG_THREADS = 512;

// Roots with 32 < k <= KM: one block per root.  Two instances: KM = TRI_KS
// for the many short lists (small shared footprint, many blocks per SM) and
// KM = TRI_KM for the long ones.
template <int KM, int THREADS, int BIN, int WORK>
__global__ void __launch_bounds__(THREADS) k_tri_block(Ctl* c, const int32_t* __restrict__ list,
                                                  const long long* __restrict__ U_off,
                                                  const uint32_t* __restrict__ U_col,
                                                  const int32_t* __restrict__ U_split,
                                                  unsigned long long* __restrict__ tpack) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    BlockTri<KM, THREADS>& S = *(BlockTri<KM, THREADS>*)smem;
    __shared__ int s_idx, s_one;
    constexpr int LG = BlockTri<KM, THREADS>::LG;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = THREADS / 32;
    const int cnt = c->nbin[BIN];
    unsigned long long ka = 0, kb = 0;
    for (;;) {
        if (tid == 0) {
            s_idx = (int)atomicAdd(&c->work[WORK], 1u);
            s_one = 0;
        }
        __syncthreads();
        const int idx = s_idx;
        if (idx >= cnt) break;
        const int32_t u = list[idx];
        const long long rb = U_off[u] + U_split[u];
        const int k = (int)(U_off[u + 1] - rb);
        const int W = (k + 31) >> 5, ws = W | 1;
        const uint32_t xmax = vid(U_col[rb + k - 1]);
        for (int j = tid; j < (1 << (LG - 5)); j += THREADS) S.bloom[j] = 0;
        for (int j = tid; j < k * ws; j += THREADS) {
            S.R[j] = 0;
            S.D[j] = 0;
        }
        for (int t = tid; t < k; t += THREADS) {
            const uint32_t x = U_col[rb + t];
            const uint32_t v = vid(x);
            const long long nb = U_off[v] + U_split[v];
            S.X[t] = x;
            S.nb[t] = nb;
            S.pre[t + 1] = (int)lower_bound_id(U_col + nb, U_off[v + 1] - nb, xmax + 1);
            S.cnt[t] = 0;
        }
        __syncthreads();
        for (int t = tid; t < k; t += THREADS) {
            const uint32_t h = tri_hash(vid(S.X[t]), LG);
            atomicOr(&S.bloom[h >> 5], 1u << (h & 31));
        }
        if (warp == 0) {  // inclusive scan of pre[1..k]
            int carry = 0;
            for (int b = 0; b < k; b += 32) {
                int x = b + lane < k ? S.pre[b + lane + 1] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    int y = __shfl_up_sync(FULL, x, o);
                    if (lane >= o) x += y;
                }
                if (b + lane < k) S.pre[b + lane + 1] = x + carry;
                carry += __shfl_sync(FULL, x, 31);
            }
            if (lane == 0) S.pre[0] = 0;
        }
        __syncthreads();
        const int total = S.pre[k];
        const Root t{S.X, S.nb, S.pre, S.bloom, S.R, S.D, S.cnt, k, ws, LG};
        int n = 0;
        bool one = false;
        for (int base = warp * 128; base < total; base += NW * 128)
            one |= tri_chunk(t, U_col, base, total, find_seg(S.pre, k, base), S.queue[warp], n, tpack);
        one |= tri_record(t, S.queue[warp], n, tpack);
        if (one) s_one = 1;
        __syncthreads();
        const bool differ = s_one != 0;
        // 4-cliques: row q against the row of each of its bits
        auto cliques = [&](int q) {
            unsigned long long x = 0;
            const uint32_t* r = S.R + q * ws;
            for (int i = 0; i < W; i++)
                for (uint32_t m = r[i]; m; m &= m - 1) {
                    const int p = i * 32 + __ffs(m) - 1;
                    const uint32_t* rp = S.R + p * ws;
                    unsigned y = 0;
                    for (int j = i; j < W; j++) y += __popc(r[j] & rp[j]);
                    x += y;
                }
            return x;
        };
        for (int q = tid; q < k; q += THREADS) {
            const uint32_t* r = S.R + q * ws;
            const uint32_t* d = S.D + q * ws;
            unsigned ta = S.cnt[q] >> 16, tb = S.cnt[q] & 0xFFFFu;
            for (int i = 0; i < W; i++) {
                ta += __popc(r[i]);
                tb += __popc(r[i] ^ d[i]);
            }
            if (ta | tb) atomicAdd(&tpack[rb + q], ((unsigned long long)ta << 32) | tb);
            const unsigned long long x = cliques(q);
            ka += x;
            if (!differ) kb += x;
        }
        if (differ) {
            __syncthreads();
            for (int j = tid; j < k * ws; j += THREADS) S.R[j] ^= S.D[j];
            __syncthreads();
            for (int q = tid; q < k; q += THREADS) kb += cliques(q);
        }
        __syncthreads();
    }
    acc_add(c, 4, ka);
    acc_add(c, 10, kb);
    stage_end(c, 4);
}

// Roots with very long out-lists: one warp per root, one lane per out-edge
// u->v merging N+(u) (after v) with N+(v); 4-cliques by a three-way merge.
__global__ void k_tri_merge(Ctl* c, const int32_t* __restrict__ list, const long long* __restrict__ U_off,
                            const uint32_t* __restrict__ U_col, const int32_t* __restrict__ U_split,
                            unsigned long long* __restrict__ tpack) {
    pdl_enter();
    const int cnt = c->nbin[BIN_TRI_MERGE];
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    unsigned long long ka = 0, kb = 0;
    for (int wi = warp; wi < cnt; wi += nwarps) {
        int32_t u = list[wi];
        long long ob = U_off[u] + U_split[u], oe = U_off[u + 1];
        for (long long e = ob + lane; e < oe; e += 32) {
            uint32_t fe = U_col[e];
            uint32_t v = vid(fe);
            long long vb = U_off[v] + U_split[v], ve = U_off[v + 1];
            long long i = e + 1, j = vb;
            while (i < oe && j < ve) {
                uint32_t ei = U_col[i], ej = U_col[j];
                uint32_t x = vid(ei), y = vid(ej);
                if (x < y) {
                    i++;
                } else if (x > y) {
                    j++;
                } else {
                    uint32_t f = fe & ei & ej;
                    unsigned long long inc = flag_inc(f);
                    if (inc) {
                        atomicAdd(&tpack[e], inc);
                        atomicAdd(&tpack[i], inc);
                        atomicAdd(&tpack[j], inc);
                        long long wb = U_off[x] + U_split[x], we = U_off[x + 1];
                        long long p = i + 1, q = j + 1, r = wb;
                        while (p < oe && q < ve && r < we) {
                            uint32_t ep = U_col[p], eq = U_col[q], er = U_col[r];
                            uint32_t a = vid(ep), b = vid(eq), cc = vid(er);
                            uint32_t mx = max(a, max(b, cc));
                            if (a == mx && b == mx && cc == mx) {
                                uint32_t g = f & ep & eq & er;
                                ka += (g & FLAG_A) ? 1 : 0;
                                kb += (g & FLAG_B) ? 1 : 0;
                                p++;
                                q++;
                                r++;
                            } else {
                                if (a < mx) p++;
                                if (b < mx) q++;
                                if (cc < mx) r++;
                            }
                        }
                    }
                    i++;
                    j++;
                }
            }
        }
    }
    acc_add(c, 4, ka);
    acc_add(c, 10, kb);
    stage_end(c, 4);
}

// ---- 4-cycles ----------------------------------------------------------------

constexpr uint32_t EMPTY_KEY = 0xFFFFFFFFu;

// packed counter: G_a count in the high 16 bits, G_b count in the low 16
__device__ __forceinline__ uint32_t flag_inc16(uint32_t f) {
    return ((f & FLAG_A) ? 0x10000u : 0u) | ((f & FLAG_B) ? 1u : 0u);
}

// open-addressing insert; returns the counter's old value
__device__ __forceinline__ uint32_t hash_add(uint32_t* keys, uint32_t* cnts, int shift, uint32_t mask, uint32_t w,
                                             uint32_t inc) {
    uint32_t h = (w * 0x9E3779B1u) >> shift;
    for (;;) {
        uint32_t k = keys[h];
        if (k == w) return atomicAdd(&cnts[h], inc);
        if (k == EMPTY_KEY) {
            uint32_t prev = atomicCAS(&keys[h], EMPTY_KEY, w);
            if (prev == EMPTY_KEY || prev == w) return atomicAdd(&cnts[h], inc);
        }
        h = (h + 1) & mask;
    }
}

__device__ __forceinline__ int log2_table(long long wt, int lo_log, int hi_log) {
    int lg = lo_log;
    while (lg < hi_log && (1ll << lg) < 2 * wt) lg++;
    return lg;
}

// w~ <= 32: every wedge endpoint in one lane; equal endpoints are grouped
// with __match_any_sync and each group adds C(c, 2).
__global__ void __launch_bounds__(256) k_c4_reg(Ctl* c, const int32_t* __restrict__ list,
                                               const long long* __restrict__ U_off,
                                               const uint32_t* __restrict__ U_col,
                                               const int32_t* __restrict__ U_split) {
    pdl_enter();
    __shared__ long long sVb[8][32];
    __shared__ uint32_t sFv[8][32];
    __shared__ int sPre[8][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int cnt = c->nbin[BIN_C4_REG];
    unsigned long long qa = 0, qb = 0, wedges = 0;
    for (int i = blockIdx.x * 8 + w; i < cnt; i += gridDim.x * 8) {
        int32_t u = list[i];
        long long rb = U_off[u];
        int nlow = U_split[u];  // 2..32 here
        int dv = 0;
        if (lane < nlow) {
            uint32_t fv = U_col[rb + lane];
            uint32_t v = vid(fv);
            long long vb = U_off[v];
            dv = (int)(U_off[v + 1] - vb);
            sVb[w][lane] = vb;
            sFv[w][lane] = fv;
        }
        int inc = dv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += y;
        }
        const int total = __shfl_sync(FULL, inc, 31);  // <= 32
        sPre[w][lane + 1] = inc;
        if (lane == 0) sPre[w][0] = 0;
        __syncwarp();
        bool ok = false;
        uint32_t wv = 0, fl = 0;
        if (lane < total) {
            int j = find_seg(sPre[w], nlow, lane);
            uint32_t e = U_col[sVb[w][j] + (lane - sPre[w][j])];
            wv = vid(e);
            ok = wv < (uint32_t)u;
            fl = sFv[w][j] & e & (FLAG_A | FLAG_B);
        }
        unsigned okm = __ballot_sync(FULL, ok);
        if (lane == 0) wedges += __popc(okm);
        bool valid = ok && fl;
        unsigned peers = __match_any_sync(FULL, valid ? wv : (0x80000000u | (uint32_t)lane));
        unsigned ba = __ballot_sync(FULL, valid && (fl & FLAG_A));
        unsigned bb = __ballot_sync(FULL, valid && (fl & FLAG_B));
        if (valid && lane == __ffs(peers) - 1) {
            qa += choose2(__popc(peers & ba));
            qb += choose2(__popc(peers & bb));
        }
        __syncwarp();
    }
    acc_add(c, 5, qa);
    acc_add(c, 11, qb);
    acc_add(c, 15, wedges);
    stage_end(c, 5);
}

// Walk the wedges u-v-w of pivot u (w < u) for its lower neighbours
// v = N(u)[j], calling fn(w, flags) once per wedge.  The warp takes 32
// lower neighbours at a time and lays their rows end to end (a warp prefix
// sum over the nonempty rows); each lane then finds its row from a bitmask
// of row starts (one OR-reduction per 32 entries), so the loads of up to 128
// entries of many short rows are in flight together instead of one row after
// the other.  Entries at or above u are read and skipped.  Rows are taken in
// groups j0 = first, first + 32 * step, ...; scratch: 32 ints, 32 int64 and
// 32 uint32 of shared memory per warp.  Warp-uniform.
constexpr int WF_UNROLL = 4;
template <class Fn>
__device__ __forceinline__ void walk_flat(const long long* __restrict__ U_off, const uint32_t* __restrict__ U_col,
                                          uint32_t u, long long rb, int nlow, int first, int step, int* cpre,
                                          long long* cvb, uint32_t* cfv, Fn fn) {
    const int lane = threadIdx.x & 31;
    for (int j0 = first * 32; j0 < nlow; j0 += step * 32) {
        const int j = j0 + lane;
        int len = 0;
        long long vb = 0;
        uint32_t fv = 0;
        if (j < nlow) {
            fv = U_col[rb + j];
            const uint32_t v = vid(fv);
            vb = U_off[v];
            len = (int)(U_off[v + 1] - vb);
        }
        const unsigned ne = __ballot_sync(FULL, len > 0);
        if (!ne) continue;
        int inc = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += y;
        }
        const int total = __shfl_sync(FULL, inc, 31);
        const int k = __popc(ne);
        __syncwarp();
        if (len > 0) {
            const int slot = __popc(ne & lanemask_lt());
            cpre[slot] = inc - len;
            cvb[slot] = vb - (inc - len);
            cfv[slot] = fv;
        }
        __syncwarp();
        const int my_start = lane < k ? cpre[lane] : 0x7FFFFFFF;
        int R = 0;  // row holding position t0 (warp-uniform)
        for (int t0 = 0; t0 < total; t0 += 32 * WF_UNROLL) {
            uint32_t ev[WF_UNROLL], fr[WF_UNROLL];
#pragma unroll
            for (int q = 0; q < WF_UNROLL; q++) {
                const int tb = t0 + q * 32;
                ev[q] = 0xFFFFFFFFu;
                fr[q] = 0;
                if (tb < total) {
                    const unsigned bit = (my_start > tb && my_start < tb + 32) ? (1u << (my_start - tb)) : 0u;
                    const unsigned m = __reduce_or_sync(FULL, bit);
                    const int r = R + __popc(m & ((2u << lane) - 1u));
                    if (tb + lane < total) {
                        ev[q] = U_col[cvb[r] + tb + lane];
                        fr[q] = cfv[r];
                    }
                    int rn = R + __popc(m);
                    if (rn + 1 < k && cpre[rn + 1] == tb + 32) rn++;
                    R = rn;
                }
            }
#pragma unroll
            for (int q = 0; q < WF_UNROLL; q++) {
                const uint32_t w = vid(ev[q]);
                if (ev[q] != 0xFFFFFFFFu && w < u) fn(w, fr[q] & ev[q] & (FLAG_A | FLAG_B));
            }
        }
        __syncwarp();
    }
}

constexpr int C4W_WARPS = 4;
constexpr int C4W_SLOTS = 2 * C4_T1;

__global__ void __launch_bounds__(C4W_WARPS * 32) k_c4_warp(Ctl* c, const int32_t* __restrict__ list,
                                                          const long long* __restrict__ U_off,
                                                          const uint32_t* __restrict__ U_col,
                                                          const int32_t* __restrict__ U_split,
                                                          const long long* __restrict__ U_wt) {
    pdl_enter();
    __shared__ uint32_t sKey[C4W_WARPS][C4W_SLOTS];
    __shared__ uint32_t sCnt[C4W_WARPS][C4W_SLOTS];
    __shared__ int s_pre[C4W_WARPS][32];
    __shared__ long long s_vb[C4W_WARPS][32];
    __shared__ uint32_t s_fv[C4W_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int cnt = c->nbin[BIN_C4_WARP];
    unsigned long long qa = 0, qb = 0, wedges = 0;
    uint32_t* keys = sKey[w];
    uint32_t* cnts = sCnt[w];
    for (int i = blockIdx.x * C4W_WARPS + w; i < cnt; i += gridDim.x * C4W_WARPS) {
        const uint32_t u = (uint32_t)list[i];
        const long long rb = U_off[u];
        const int nlow = U_split[u];
        const int lg = log2_table(U_wt[u], 5, 10);
        const uint32_t mask = (1u << lg) - 1;
        const int shift = 32 - lg;
        for (int s = lane; s <= (int)mask; s += 32) {
            keys[s] = EMPTY_KEY;
            cnts[s] = 0;
        }
        __syncwarp();
        walk_flat(U_off, U_col, u, rb, nlow, 0, 1, s_pre[w], s_vb[w], s_fv[w], [&](uint32_t wv, uint32_t fl) {
            wedges++;
            if (!fl) return;
            uint32_t old = hash_add(keys, cnts, shift, mask, wv, flag_inc16(fl));
            if (fl & FLAG_A) qa += old >> 16;
            if (fl & FLAG_B) qb += old & 0xFFFFu;
        });
        __syncwarp();
    }
    acc_add(c, 5, qa);
    acc_add(c, 11, qb);
    acc_add(c, 15, wedges);
    stage_end(c, 5);
}

// ---- per-edge terms and closed forms ----------------------------------------

constexpr int ET_WARPS = 8;
constexpr int ET_LONG = 256;  // longer out-lists are walked one at a time
struct EdgeRow {
    long long b;      // first entry of the out-list
    int k;            // its length
    uint32_t da, db;  // degrees in G_a, G_b
};
// Bound by latency: two random degree loads per edge behind a chain of three.
// A warp takes 32 vertices and walks their out-lists as one run, four edges a
// lane ahead, so rows of a few entries fill the lanes (a warp per row: 3.25 ms
// for the 69 M edges of a 4.8 M-vertex graph, 0.60 now).  The sums meet in the
// block before the atomics (a 7,000-vertex graph: 14 us with a set per warp,
// now 9).
__global__ void __launch_bounds__(ET_WARPS * 32, 4)
    k_edge_terms(Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                 const uint32_t* __restrict__ U_col, const int32_t* __restrict__ U_split,
                 const unsigned long long* __restrict__ tpack, const int32_t* __restrict__ da,
                 const int32_t* __restrict__ db) {
    pdl_enter();
    __shared__ EdgeRow s_row[ET_WARPS * 32];
    __shared__ int s_pre[ET_WARPS][33];
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = (gridDim.x * blockDim.x) >> 5;
    EdgeRow* const rows = s_row + (threadIdx.x & ~31);
    int* const pre = s_pre[threadIdx.x >> 5];
    unsigned long long P[2] = {0, 0}, S[2] = {0, 0}, T[2] = {0, 0}, D[2] = {0, 0}, work = 0;
    unsigned long long T3[2] = {0, 0}, W2[2] = {0, 0};  // sum of t_e; sum of C(d, 2)
    unsigned E[2] = {0, 0};
    auto edge = [&](const EdgeRow& r, uint32_t fe, unsigned long long t, uint32_t dva, uint32_t dvb) {
        auto add = [&](int g, uint32_t du, uint32_t dv, uint32_t tt) {
            P[g] += (unsigned long long)(du - 1) * (dv - 1);
            T[g] += (unsigned long long)tt * (du + dv - 4);  // (an edge in a triangle has du, dv >= 2)
            D[g] += (unsigned long long)tt * tt;
            T3[g] += tt;
            E[g]++;
        };
        if (fe & FLAG_A) add(0, r.da, dva, (uint32_t)(t >> 32));
        if (fe & FLAG_B) add(1, r.db, dvb, (uint32_t)t);
    };
    const int quads = (nW + 3) / 4;
    // eight quads of neighbouring vertices, spread over the ids (hubs have
    // neighbouring ids)
    for (long long base = warp; base < quads; base += 8 * nwarps) {
        const long long i = 4 * (base + (lane >> 2) * nwarps) + (lane & 3);
        EdgeRow r{};
        if (i < nW) {
            const int32_t u = wlist[i];
            r.da = (uint32_t)da[u];
            r.db = (uint32_t)db[u];
            S[0] += choose3(r.da);
            S[1] += choose3(r.db);
            W2[0] += choose2(r.da);
            W2[1] += choose2(r.db);
            const long long b = U_off[u], e = U_off[u + 1];
            r.b = b + U_split[u];
            r.k = (int)(e - r.b);
            // rows walked for the triangles: both out-lists of every edge, so
            // a vertex's own once for each of its edges
            work += (unsigned long long)r.k * (unsigned long long)(e - b);
        }
        const bool is_long = r.k > ET_LONG;
        rows[lane] = r;
        int x = is_long ? 0 : r.k;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        pre[lane + 1] = x;
        if (lane == 0) pre[0] = 0;
        const int total = __shfl_sync(FULL, x, 31);
        __syncwarp();
        int q = 0;
        for (int j0 = lane; j0 < total; j0 += 128) {
            int at[4];
            uint32_t fe[4], va[4], vb[4];
            unsigned long long t[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int j = j0 + 32 * k;
                if (j < total)
                    while (pre[q + 1] <= j) q++;
                at[k] = q;
                const long long e = rows[q].b + (j - pre[q]);
                fe[k] = j < total ? U_col[e] : 0u;
                t[k] = j < total ? tpack[e] : 0ull;
            }
#pragma unroll
            for (int k = 0; k < 4; k++) {
                va[k] = (fe[k] & FLAG_A) ? (uint32_t)da[vid(fe[k])] : 0u;
                vb[k] = (fe[k] & FLAG_B) ? (uint32_t)db[vid(fe[k])] : 0u;
            }
#pragma unroll
            for (int k = 0; k < 4; k++) edge(rows[at[k]], fe[k], t[k], va[k], vb[k]);
        }
        for (unsigned m = __ballot_sync(FULL, is_long); m; m &= m - 1) {
            const EdgeRow l = rows[__ffs(m) - 1];
#pragma unroll 4
            for (int j = lane; j < l.k; j += 32) {
                const uint32_t fe = U_col[l.b + j];
                edge(l, fe, tpack[l.b + j], (fe & FLAG_A) ? (uint32_t)da[vid(fe)] : 0u,
                     (fe & FLAG_B) ? (uint32_t)db[vid(fe)] : 0u);
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int g = 0; g < 2; g++) {
        P[g] -= T3[g];             // sum of (du - 1)(dv - 1) - t
        D[g] = (D[g] - T3[g]) / 2;  // sum of C(t, 2), exact: every term is even
    }
    // one atomic per sum and block
    __shared__ unsigned long long s_sum[ET_WARPS][NACC];
    unsigned long long* const mine = s_sum[threadIdx.x >> 5];
    if (lane < NACC) mine[lane] = 0;
    __syncwarp();
    auto put = [&](int slot, unsigned long long x) {
        x = warp_sum_u64(x);
        if (lane == 0) mine[slot] = x;
    };
    if (warp < quads) {
#pragma unroll
        for (int g = 0; g < 2; g++) {
            put(6 * g + 0, P[g]);
            put(6 * g + 1, S[g]);
            put(6 * g + 2, T[g]);
            put(6 * g + 3, D[g]);
            put(12 + g, E[g]);
            put(16 + g, T3[g]);
            put(18 + g, W2[g]);
        }
        put(14, work);
    }
    __syncthreads();
    if (threadIdx.x < NACC) {
        unsigned long long x = 0;
        for (int w = 0; w < ET_WARPS; w++) x += s_sum[w][threadIdx.x];
        if (x) atomicAdd(&c->accs[threadIdx.x][blockIdx.x & (ACC_STRIPES - 1)], x);
    }
}

// The closed forms and the results, by one warp (lane i < 6 holds graphlet i,
// so the loads of one result are in flight together).
// mode 0: committed batch, F += C_a - C_b (unless the batch was rejected);
// mode 2: independent batch, the result is F + C_a - C_b and F stays; mode 1:
// static count; mode 3: a committed batch whose pass covered every vertex, so
// C_a and C_b are the whole graph's counts after and before it: F = C_a, and
// C_b is the result of the batch before it (committed without a count of its
// own); mode 4: two independent batches counted over every vertex (the twin
// pass): C_a and C_b are the whole graph's counts with the first and with the
// second batch applied; F stays
__global__ void k_finalize(Ctl* c, int mode) {
    pdl_enter();
    __shared__ unsigned long long s_acc[32];
    const int t = threadIdx.x;
    if (blockIdx.x != 0 || t >= 32) return;
    const bool ok = c->err == 0 && c->active;
    unsigned long long x = 0;  // fold the striped accumulators
    if (t < NACC) {
        x = c->acc[t];
#pragma unroll
        for (int k = 0; k < ACC_STRIPES; k++) x += c->accs[t][k];
        c->acc[t] = x;
    }
    s_acc[t] = x;
    const unsigned long long F = t < 6 ? c->F[t] : 0ull, F3 = t < 2 ? c->F3[t] : 0ull;
    __syncwarp();
    long long C[2] = {0, 0};
    for (int g = 0; g < 2; g++) {
        const unsigned long long* s = s_acc + 6 * g;
        const long long P = (long long)s[0], S = (long long)s[1], TT = (long long)(s[2] / 2), D = (long long)s[3],
                        K = (long long)s[4], Q = (long long)s[5];
        const long long g6 = K;
        const long long g5 = D - 6 * K;
        const long long g3 = Q - g5 - 3 * K;
        const long long g4 = TT - 4 * g5 - 12 * K;
        const long long g2 = S - g4 - 2 * g5 - 4 * K;
        const long long g1 = P - 2 * g4 - 4 * g3 - 6 * g5 - 12 * K;
        C[g] = t == 0 ? g1 : t == 1 ? g2 : t == 2 ? g3 : t == 3 ? g4 : t == 4 ? g5 : g6;
        if (t < 6) {
            (g == 0 ? c->Ca : c->Cb)[t] = C[g];
            (g == 0 ? c->sa : c->sb)[t] = t == 0 ? P : t == 1 ? S : t == 2 ? TT : t == 3 ? D : t == 4 ? K : Q;
        }
    }
    if (t < 6) {
        const unsigned long long d = (unsigned long long)(C[0] - C[1]);
        unsigned long long f = F;
        if (mode == 0 && ok) f = F + d;
        if (mode == 3 && ok) {
            c->prev_out[t] = (unsigned long long)C[1];
            f = (unsigned long long)C[0];
        }
        if (f != F) c->F[t] = f;
        c->last_out[t] = mode == 2 ? F + d : mode == 4 ? (unsigned long long)C[0] : f;
        if (mode == 4) c->prev_out[t] = (unsigned long long)C[1];
    }
    // 3-vertex graphlets from the same sums: triangles = (sum t_e) / 3,
    // induced 2-paths = sum C(d, 2) - 3 triangles
    if (t < 2) {
        long long C3[2];
        for (int g = 0; g < 2; g++) {
            const unsigned long long t3 = s_acc[16 + g], w2 = s_acc[18 + g];
            C3[g] = t == 0 ? (long long)(w2 - t3) : (long long)(t3 / 3);
            (g == 0 ? c->C3a : c->C3b)[t] = C3[g];
        }
        const unsigned long long d = (unsigned long long)(C3[0] - C3[1]);
        unsigned long long f = F3;
        if (mode == 0 && ok) f = F3 + d;
        if (mode == 3 && ok) f = (unsigned long long)C3[0];
        if (f != F3) c->F3[t] = f;
        c->last_out3[t] = mode == 2 ? F3 + d : f;
    }
    if (t == 0) c->ts[6] = global_ns();
}

}  // namespace gcx

// ---- launch sequence of one counting pass -------------------------------------

namespace gcx {

void count_setup_attributes() {
    cudaFuncSetAttribute(k_tri_block<TRI_KM, TRI_BIG_THREADS, BIN_TRI_BLOCK, WORK_TRI_BLOCK>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BlockTri<TRI_KM, TRI_BIG_THREADS>));
    cudaFuncSetAttribute(k_tri_block<TRI_KS, TRI_SMALL_THREADS, BIN_TRI_SMALL, WORK_TRI_SMALL>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(BlockTri<TRI_KS, TRI_SMALL_THREADS>));
    c4_setup_attributes();
}

// The caller's bin boundaries, clamped to what the kernels and the scratch
// of this pass can take.
Tuning effective_tuning(const CountArgs& a) {
    Tuning t = a.tune;
    t.tri_warp_max = std::max(1, std::min(t.tri_warp_max, 32));
    t.tri_small_max = std::max(t.tri_warp_max, std::min(t.tri_small_max, TRI_KS));
    t.tri_block_max = std::max(t.tri_small_max, std::min(t.tri_block_max, TRI_KM));
    t.c4_reg_max = std::max(1, std::min(t.c4_reg_max, 32));
    t.c4_warp_max = std::max(t.c4_reg_max, std::min(t.c4_warp_max, C4_T1));
    t.c4_block_max = std::max(t.c4_warp_max, std::min(t.c4_block_max, C4_T2));
    t.c4_cta_max = std::max<long long>(t.c4_block_max, std::min<long long>(t.c4_cta_max, C4_T3));
    return t;
}

int enqueue_counting(const CountArgs& a, cudaStream_t s, int mode) {
    const int sms = a.sms;
    int nl = 0;
    auto lists = [&](int b) { return a.bins + (size_t)b * a.n_alloc; };
    long long nw = a.n_alloc > 0 ? a.n_alloc : 1;
    int gb = (int)std::min<long long>((nw + 255) / 256, 8LL * sms);
    Tuning t = effective_tuning(a);
    if (a.c4_mode != C4_COUNT && a.local_heavy_min > 0) {
        const long long cap = std::max<long long>(1, a.local_heavy_min - 1);
        t.c4_reg_max = (int)std::min<long long>(t.c4_reg_max, cap);
        t.c4_warp_max = (int)std::min<long long>(t.c4_warp_max, cap);
        t.c4_block_max = (int)std::min<long long>(t.c4_block_max, cap);
        t.c4_cta_max = std::min(t.c4_cta_max, cap);
    }
    // The triangle kernels and the 4-cycle tiers are independent: with
    // auxiliary streams they run side by side in six branches (4-cycle warps on
    // the handle's own stream; triangle warp roots; block roots; small tables;
    // larger tables; pivots) between a fork after the binning and a join before
    // the edge terms.  On a small graph each branch is a few kernels bound by
    // latency, and the count takes the longest branch.  The pivots' plan and
    // run bounds need the sums of k_wedge_bound only and run beside the
    // binning; after it they would wait until the triangle kernels, which fill
    // the chip, let go of a first SM (20 us of a 7,000-vertex graph's batch).
    bool par = true;
    for (int i = 0; i < NAUX; i++) par = par && a.aux[i];
    cudaStream_t sT = par ? a.aux[0] : s, sB = par ? a.aux[1] : s, sC = par ? a.aux[2] : s,
                 sD = par ? a.aux[3] : s, sP = par ? a.aux[4] : s;
    PivotArgs pa;
    pa.ctl = a.ctl;
    pa.pivots = lists(BIN_C4_DENSE);
    pa.U_off = a.U_off;
    pa.U_col = a.U_col;
    pa.U_split = a.U_split;
    pa.U_wt = a.U_wt;
    pa.n = a.n_alloc;
    pa.b = a.c4;
    const C4Geom geom = c4_geom(a.n_alloc, sms);
    pa.words = geom.words;
    pa.group = geom.group;
    pa.credit = a.c4_credit;
    pdl_launch(k_wedge_bound, dim3(8 * sms), dim3(256), 0, s, a.ctl, a.wlist, a.U_off, a.U_col, a.U_split, a.U_wt, t);
    if (par) {
        cudaEventRecord(a.fork, s);
        cudaStreamWaitEvent(sP, a.fork, 0);
    }
    nl += enqueue_c4_plan(pa, geom, sP);
    pdl_launch(k_bin, dim3(gb), dim3(256), 0, s, a.ctl, a.wlist, a.U_off, a.U_split, a.U_wt, a.bins, a.n_alloc, t);
    nl += 2;
    if (par) {
        cudaEventRecord(a.fork, s);
        for (int i = 0; i < NAUX; i++) cudaStreamWaitEvent(a.aux[i], a.fork, 0);
    }
    nl += enqueue_c4_pivots(pa, a.c4_mode, geom, sP);
    k_tri_warp<<<4 * sms, TW * 32, 0, sT>>>(a.ctl, lists(BIN_TRI_WARP), a.U_off, a.U_col, a.U_split, a.tpack);
    k_tri_block<TRI_KS, TRI_SMALL_THREADS, BIN_TRI_SMALL, WORK_TRI_SMALL>
        <<<8 * sms, TRI_SMALL_THREADS, sizeof(BlockTri<TRI_KS, TRI_SMALL_THREADS>), sB>>>(
            a.ctl, lists(BIN_TRI_SMALL), a.U_off, a.U_col, a.U_split, a.tpack);
    k_tri_block<TRI_KM, TRI_BIG_THREADS, BIN_TRI_BLOCK, WORK_TRI_BLOCK>
        <<<2 * sms, TRI_BIG_THREADS, sizeof(BlockTri<TRI_KM, TRI_BIG_THREADS>), sB>>>(
            a.ctl, lists(BIN_TRI_BLOCK), a.U_off, a.U_col, a.U_split, a.tpack);
    k_tri_merge<<<sms, 256, 0, sB>>>(a.ctl, lists(BIN_TRI_MERGE), a.U_off, a.U_col, a.U_split, a.tpack);
    nl += 4;
    if (a.c4_mode == C4_COUNT) {
        k_c4_reg<<<4 * sms, 256, 0, s>>>(a.ctl, lists(BIN_C4_REG), a.U_off, a.U_col, a.U_split);
        k_c4_warp<<<7 * sms, C4W_WARPS * 32, 0, s>>>(a.ctl, lists(BIN_C4_WARP), a.U_off, a.U_col, a.U_split,
                                                      a.U_wt);
        nl += 2;
    } else {
        nl += enqueue_c4_warp_credit(pa, a.c4_mode, a.bins, sms, s);
    }
    nl += enqueue_c4_tables(pa, a.c4_mode, a.bins, sms, sC, sD);
    if (par)
        for (int i = 0; i < NAUX; i++) {
            cudaEventRecord(a.join[i], a.aux[i]);
            cudaStreamWaitEvent(s, a.join[i], 0);
        }
    k_edge_terms<<<8 * sms, ET_WARPS * 32, 0, s>>>(a.ctl, a.wlist, a.U_off, a.U_col, a.U_split, a.tpack, a.da, a.db);
    pdl_launch(k_finalize, dim3(1), dim3(32), 0, s, a.ctl, mode);
    nl += 2;
    return nl;
}

}  // namespace gcx
