// gc_cycles.cu -- 4-cycles of the pivots beyond the warp tier: the wedges of a
// pivot counted in shared memory, for the global counts and, with a second
// walk that credits what was counted, per vertex and per edge.
//
// A pivot u needs c_w = #{v in N(u) n N(w): v, w < u} for every w below it
// (gc_count.cu): one counter increment per wedge u-v-w, and sum C(c_w, 2) is
// the sum of the old values that the increments return.  L2 atomics top out
// near 130 G/s on this chip, shared-memory ones near 1.8 T/s.
//
// Small and medium pivots (k_c4_table): a block's hash table holds every
// endpoint, so a pivot is one task.
//
// Large pivots (k_c4_pivot): the ids are cut into chunks whose counters fill
// one block's shared array, and a block takes one (chunk, pivot) at a time:
// rows are sorted, so the part of a lower neighbour's row that lies in a
// chunk is one contiguous run, and the chunks of a pivot need not meet.
//  * Counter width.  c_w is at most the degree of w, and ids ascend with the
//    initial degree, so most chunks need few bits: 4, 8, 16 or 32 per counter,
//    chosen from the largest union-graph degree in the chunk (k_c4_granules,
//    k_c4_plan).  A graph of 1.6 M vertices and 30 M edges takes 7 chunks
//    instead of the 33 of 32-bit counters.
//  * Run bounds.  k_c4_runs writes, for each chunk and vertex, the start and
//    length of the vertex's run in one 8-byte word, so a lower neighbour costs
//    one random load per chunk.  At most `group` chunks are held at a time;
//    graphs with more chunks take more (runs, pivots) launches.
//  * Order.  Tasks run chunk by chunk, so the runs and adjacency entries of one
//    chunk (a few tens of MB) stay in L2 while every pivot walks them, and from
//    the pivot of most wedges down.
//  * Two graphs.  A wedge in both graphs counts in the shared counters.  The
//    few in one graph only (through a changed pair) are listed; after the
//    increments each adds the both-graph count of its endpoint (the cross
//    term of C(c_ab + c_x, 2)), and then the list of each graph runs through
//    the cleared counters by itself.
//
// Local counts.  A 4-cycle through pivot u and opposite corner w credits u,
// w and its two middle vertices (or its four edges).  Once a task's c_w are
// known, a second walk adds c_w - 1 to each middle vertex (to both edges of
// each wedge), and the sweep that clears the counters adds C(c_w, 2) to w.
// On the 1.6M/30M graph the pivots take 24 ms with the credits per vertex, 11.7
// without; 33.5 when the sweep looked at every counter of a word and runs were
// summed by shuffles.
#include <algorithm>

#include "gc_c4.cuh"
#include "gc_kernels.cuh"
#include "gc_walk.cuh"

namespace gcx {

namespace {

constexpr unsigned long long RUN_LEN = (1ull << 28) - 1;
constexpr int C4_SPLITS = 18;  // chunks that the share limit may add

__device__ __forceinline__ void red_u64(unsigned long long* p, unsigned long long x) { atomicAdd(p, x); }

}  // namespace

// Largest union-graph degree of each granule of `gran` consecutive ids.
__global__ void __launch_bounds__(256) k_c4_granules(const long long* __restrict__ U_off, int n, int gran,
                                                     int32_t* __restrict__ gmax) {
    pdl_enter();
    __shared__ int s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    const long long lo = (long long)blockIdx.x * gran, hi = min((long long)n, lo + gran);
    int m = 0;
    for (long long v = lo + threadIdx.x; v < hi; v += blockDim.x) m = max(m, (int)(U_off[v + 1] - U_off[v]));
    m = __reduce_max_sync(FULL, m);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, m);
    __syncthreads();
    if (threadIdx.x == 0) gmax[blockIdx.x] = s_max;
}

// Cut [0, n) into chunks, from the highest granule down: a chunk grows while
// its counters fit `words` and its share of the adjacency entries is within
// the limit.  The limit is 1 unless the pivot of most wedges would outlast an
// even share of all of them over the blocks.  One block.  Below 2^16 ids all
// counters fit at 16 bits, and the cuts are those of even shares, found by a
// thread per granule; else the walk over the granules (at most a few hundred
// on graphs below 16 M vertices) is serial.
constexpr int PLAN_TILE = 512;
__global__ void __launch_bounds__(PLAN_TILE) k_c4_plan(Ctl* c, const long long* __restrict__ U_off, int n,
                                                       int gran, int ngran, const int32_t* __restrict__ gmax,
                                                       int words, int ctas, int nchmax, C4Head* __restrict__ head,
                                                       C4Chunk* __restrict__ chunk) {
    stage_begin(c, 8);
    __shared__ int s_max[PLAN_TILE];
    __shared__ long long s_off[PLAN_TILE + 1];
    const long long entries = U_off[n];
    if (c->c4_wt == 0 || entries == 0) {  // no pivots
        if (threadIdx.x == 0) head->nch = 0;
        return;
    }
    int nch = 0, hi = n, lo = n, cmax = 0, cs = 3;
    long long cmass = 0, limit = entries;
    {
        const double fair = (double)c->c4_wt / ctas, big = 2.0 * (double)c->c4_wmax;
        if (big > fair) limit = max(1ll, (long long)((double)entries * fmax(fair / big, 0.125)));
    }
    if (!gmax) {
        const int t = threadIdx.x, k = (int)((entries + limit - 1) / limit);
        auto off = [&](int j) { return U_off[min((long long)n, (long long)j * gran)]; };
        auto part = [&](int j) { return (int)((entries - off(j + 1)) * k / entries); };  // of granule j
        // granule t is the highest of its chunk
        const bool cut = t < ngran && (t == ngran - 1 || part(t) != part(t + 1));
        const unsigned b = __ballot_sync(FULL, cut);
        __shared__ unsigned s_cut[PLAN_TILE / 32];
        __shared__ int s_top[PLAN_TILE];
        if ((t & 31) == 0) s_cut[t >> 5] = b;
        __syncthreads();
        int at = __popc(b & ~(lanemask_lt() | (1u << (t & 31)))), all = 0;
        for (int w = 0; w < PLAN_TILE / 32; w++) {
            all += __popc(s_cut[w]);
            if (w > (t >> 5)) at += __popc(s_cut[w]);
        }
        if (cut) s_top[at] = t + 1;
        __syncthreads();
        if (t < all && t < nchmax) {
            const int hi = s_top[t], lo = t + 1 < all ? s_top[t + 1] : 0;
            chunk[t] = C4Chunk{lo * gran, min(n, hi * gran), 1, (float)((double)(off(hi) - off(lo)) / (double)entries)};
        }
        if (t == 0) head->nch = min(all, nchmax);
        return;
    }
    for (int top = ngran; top > 0; top -= PLAN_TILE) {
        const int base = max(0, top - PLAN_TILE), cnt = top - base;
        __syncthreads();
        for (int i = threadIdx.x; i <= cnt; i += blockDim.x) {
            s_off[i] = U_off[min((long long)n, (long long)(base + i) * gran)];
            if (i < cnt) s_max[i] = gmax[base + i];
        }
        __syncthreads();
        if (threadIdx.x != 0) continue;
        for (int i = cnt - 1; i >= 0; i--) {
            const int glo = (base + i) * gran;
            const long long gm = s_off[i + 1] - s_off[i];
            const int nm = max(cmax, s_max[i]);
            const int ns = nm <= 15 ? 3 : nm <= 255 ? 2 : nm <= 65535 ? 1 : 0;
            if (lo < hi && ((long long)(hi - glo) > ((long long)words << ns) || cmass + gm > limit)) {
                if (nch < nchmax) chunk[nch++] = C4Chunk{lo, hi, cs, (float)((double)cmass / (double)entries)};
                hi = lo;
                cmax = s_max[i];
                cmass = gm;
                cs = cmax <= 15 ? 3 : cmax <= 255 ? 2 : cmax <= 65535 ? 1 : 0;
            } else {
                cmax = nm;
                cs = ns;
                cmass += gm;
            }
            lo = glo;
        }
    }
    if (threadIdx.x == 0) {
        if (lo < hi && nch < nchmax) chunk[nch++] = C4Chunk{lo, hi, cs, (float)((double)cmass / (double)entries)};
        head->nch = nch;
    }
}

// Run of every vertex's row in the chunks [c0, c0 + group): start << 28 |
// length.  A thread per vertex, chunks from the top, each bound a binary
// search in what is left of the row; where the launch has a thread for each
// (chunk, vertex), each finds its two bounds by itself (7,000 vertices:
// 16 us -> 7, all of it the latency of the searches).
__global__ void __launch_bounds__(256) k_c4_runs(const long long* __restrict__ U_off,
                                                 const uint32_t* __restrict__ U_col, int n, C4Head* __restrict__ head,
                                                 const C4Chunk* __restrict__ chunk, int c0, int group,
                                                 unsigned long long* __restrict__ run) {
    pdl_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0) head->task = 0;
    const int nc = min(group, head->nch - c0);
    if (nc <= 0) return;
    if ((long long)n * nc <= (long long)gridDim.x * blockDim.x) {
        const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
        if (i >= (long long)n * nc) return;
        const int k = (int)(i / n);
        const long long v = i - (long long)k * n, b = U_off[v], len = U_off[v + 1] - b;
        const int lo = chunk[c0 + k].lo, hi = chunk[c0 + k].hi;
        const long long s = (len && lo) ? lower_bound_id(U_col + b, len, (uint32_t)lo) : 0;
        const long long e = (len && hi < n) ? lower_bound_id(U_col + b, len, (uint32_t)hi) : len;
        run[(size_t)k * n + v] = ((unsigned long long)(b + s) << 28) | (unsigned long long)(e - s);
        return;
    }
    const int top = chunk[c0].hi;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
         v += (long long)gridDim.x * blockDim.x) {
        const long long b = U_off[v];
        long long len = U_off[v + 1] - b;
        if (len && top < n) len = lower_bound_id(U_col + b, len, (uint32_t)top);
        for (int k = 0; k < nc; k++) {
            const int lo = chunk[c0 + k].lo;
            const long long s = (len && lo) ? lower_bound_id(U_col + b, len, (uint32_t)lo) : 0;
            run[(size_t)k * n + v] = ((unsigned long long)(b + s) << 28) | (unsigned long long)(len - s);
            len = s;
        }
    }
}

// The task that a block works on, fetched while the one before it runs.
struct C4Task {
    unsigned long long id;
    long long rb;
    uint32_t u;
    int k, nlow;
    float wt;
};

// The lowest bit of each of the word's counters (32 >> s bits) that is 2 or more.
__device__ __forceinline__ uint32_t counters_above_1(uint32_t w, int s) {
    return s == 3   ? ((w >> 1) | (w >> 2) | (w >> 3)) & 0x11111111u
           : s == 2 ? __vcmpgtu4(w, 0x01010101u) & 0x01010101u
           : s == 1 ? __vcmpgtu2(w, 0x00010001u) & 0x00010001u
                    : (w > 1 ? 1u : 0u);
}

// The pivots of BIN_C4_DENSE, a block per (chunk, pivot).  Bound by issue
// slots (78 instructions per 32 wedges, 68 % of the cycles issue) and by the
// chain of three loads that starts each group of lower neighbours.  The
// counters are cleared by a fill, or, when the task has few wedges for its
// counters, by walking them again.  MODE: C4_COUNT, C4_VERTEX or C4_EDGE
// (credits; every entry is then in both graphs).
// Measured (pivots above w~ = 19,456, kernel alone): 11.7 ms for 2.85e9 wedges
// of the 1.6M/30M graph, where L2 reductions by clusters of eight blocks took
// 30 ms; 2.8 ms against 11 for 1.09e9 wedges of the 2.4M/5M graph with hubs of
// 40,000; 35 ms against 75 on the 4.8M/69M graph.
template <int MODE, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) k_c4_pivot(PivotArgs a, int c0) {
    pdl_enter();
    extern __shared__ __align__(16) uint32_t sm[];
    constexpr int NW = THREADS / 32;
    uint32_t* const cnt = sm;
    __shared__ C4Task s_task[2];
    __shared__ int s_grp[2];
    __shared__ unsigned s_nl[2];  // listed wedges of even / odd tasks
    const int tid = threadIdx.x, warp = tid >> 5;
    WarpRuns& W = ((WarpRuns*)(sm + a.words))[warp];
    const int nc = min(a.group, a.b.head->nch - c0);
    const int npiv = a.ctl->nbin[BIN_C4_DENSE];
    if (nc <= 0 || npiv == 0) return;
    const unsigned long long tasks = (unsigned long long)nc * (unsigned)npiv;
    uint32_t* const lst = a.b.list + (size_t)blockIdx.x * a.b.lcap;
    uint4* const c4 = (uint4*)cnt;
    for (int i = tid; i < a.words / 4; i += THREADS) c4[i] = make_uint4(0, 0, 0, 0);
    auto fetch = [&](C4Task& o) {
        o.id = atomicAdd(&a.b.head->task, 1ull);
        if (o.id >= tasks) return;
        o.k = (int)(o.id / (unsigned)npiv);
        o.u = (uint32_t)a.pivots[(int)(o.id - (unsigned long long)o.k * (unsigned)npiv)];
        o.rb = a.U_off[o.u];
        o.nlow = a.U_split[o.u];
        o.wt = (float)a.U_wt[o.u];
    };
    if (tid == 0) {
        fetch(s_task[0]);
        s_grp[0] = 0;
        s_nl[0] = 0;
    }
    unsigned long long qa = 0, qb = 0, qab = 0, wedges = 0;
    auto norow = [](unsigned long long, uint32_t, int) {};
    __syncthreads();
    for (int it = 0;; it++) {
        const C4Task t = s_task[it & 1];
        if (t.id >= tasks) break;
        const C4Chunk ck = a.b.chunk[c0 + t.k];
        const uint32_t lo = (uint32_t)ck.lo, u = t.u, lim = u - lo;
        const int s = ck.s, ls = 5 - s, used = (ck.hi - ck.lo + (1 << s) - 1) >> s;
        const uint32_t sub = (1u << s) - 1, cmask = 0xFFFFFFFFu >> (32 - (32 >> s));
        const int nlow = lo < u ? t.nlow : 0;
        const uint32_t* const row = a.U_col + t.rb;
        const unsigned long long* const runs = a.b.run + (size_t)t.k * a.n;
        const float est = t.wt * ck.share;  // wedges of this task, about
        const Deal deal = deal_groups(nlow, est, NW);
        auto run = [&](uint32_t fv, const uint32_t** p, int* len) {
            const unsigned long long r = runs[vid(fv)];
            *len = (int)(r & RUN_LEN);
            *p = a.U_col + (r >> 28);
        };
        auto each4 = [&](const uint32_t* const(&q)[PV_UNROLL], const uint32_t(&e)[PV_UNROLL],
                         const uint32_t(&f)[PV_UNROLL], auto one) {
#pragma unroll
            for (int i = 0; i < PV_UNROLL; i++) {
                const uint32_t x = vid(e[i]) - lo;
                if (q[i] && x < lim) one(x, e[i] & f[i]);
            }
        };
        if (tid == 0) {
            s_grp[1] = 0;
            s_nl[(it + 1) & 1] = 0;
        }
        if (tid == THREADS - 1) fetch(s_task[(it + 1) & 1]);
        unsigned long long old = 0;
        walk_lower<false>(row, nlow, deal, &s_grp[0], W, run,
                          [&](const auto& q, const auto& e, const auto& f, auto&) {
                              each4(q, e, f, [&](uint32_t x, uint32_t both) {
                                  wedges++;
                                  const uint32_t sh = (x & sub) << ls;
                                  if (both >= (FLAG_A | FLAG_B)) {
                                      old += (atomicAdd(&cnt[x >> s], 1u << sh) >> sh) & cmask;
                                  } else if (MODE == C4_COUNT && both >> 30) {
                                      const unsigned at = atomicAdd(&s_nl[it & 1], 1u);
                                      if (at < a.b.lcap) lst[at] = x | (both & FLAG_B);
                                  }
                              });
                          },
                          norow);
        qab += old;
        __syncthreads();
        if (tid == 0) s_grp[0] = 0;
        if (MODE != C4_COUNT) {
            if (MODE == C4_VERTEX) {
                old = warp_sum_u64(old);
                if ((tid & 31) == 0 && old) red_u64(&a.credit[u], old);
            }
            walk_lower<true>(
                row, nlow, deal, &s_grp[1], W, run,
                [&](const auto& q, const auto& e, const auto&, auto& x) {
#pragma unroll
                    for (int i = 0; i < PV_UNROLL; i++) {
                        const uint32_t y = vid(e[i]) - lo;
                        x[i] = 0;
                        if (q[i] && y < lim) {
                            x[i] = ((cnt[y >> s] >> ((y & sub) << ls)) & cmask) - 1;
                            if (MODE == C4_EDGE && x[i]) red_u64(&a.credit[q[i] - a.U_col], x[i]);
                        }
                    }
                },
                [&](unsigned long long sum, uint32_t fv, int j) {
                    red_u64(&a.credit[MODE == C4_EDGE ? (size_t)(t.rb + j) : (size_t)vid(fv)], sum);
                });
            __syncthreads();
            if (MODE == C4_EDGE) {
                for (int i = tid; i < (used + 3) / 4; i += THREADS) c4[i] = make_uint4(0, 0, 0, 0);
            } else {
                // C(c, 2) to every id counted twice or more
                for (int i = tid; i < (used + 3) / 4; i += THREADS) {
                    const uint4 v = c4[i];
                    if (!(v.x | v.y | v.z | v.w)) continue;
                    c4[i] = make_uint4(0, 0, 0, 0);
                    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        for (uint32_t m = counters_above_1(w4[k], s); m; m &= m - 1) {
                            const int sh = __ffs(m) - 1;
                            const unsigned long long c = (w4[k] >> sh) & cmask;
                            red_u64(&a.credit[lo + ((uint32_t)(4 * i + k) << s) + (sh >> ls)], c * (c - 1) / 2);
                        }
                }
            }
            __syncthreads();
            continue;
        }
        const unsigned nl = s_nl[it & 1];
        if (nl) {
            // Wedges in one graph only.  each(fn) runs fn(x, in_b) for each of
            // them: from the list, or, if it overflowed, by walking again
            // (ends with a barrier).
            auto each = [&](auto fn) {
                if (nl <= a.b.lcap) {
                    for (unsigned i = tid; i < nl; i += THREADS) {
                        const uint32_t e = lst[i];
                        fn(e & 0x7FFFFFFFu, (e >> 31) != 0);
                    }
                } else {
                    walk_lower<false>(row, nlow, deal, &s_grp[1], W, run,
                                      [&](const auto& q, const auto& e, const auto& f, auto&) {
                                          each4(q, e, f, [&](uint32_t x, uint32_t both) {
                                              const uint32_t g = both >> 30;
                                              if (g == 1u || g == 2u) fn(x, g == 2u);
                                          });
                                      },
                                      norow);
                    __syncthreads();
                    if (tid == 0) s_grp[1] = 0;
                }
                __syncthreads();
            };
            each([&](uint32_t x, bool in_b) {
                const unsigned c = (cnt[x >> s] >> ((x & sub) << ls)) & cmask;
                if (in_b) qb += c;
                else qa += c;
            });
            for (int i = tid; i < (used + 3) / 4; i += THREADS) c4[i] = make_uint4(0, 0, 0, 0);
            __syncthreads();
            for (int g = 0; g < 2; g++) {
                each([&](uint32_t x, bool in_b) {
                    if (in_b != (g == 1)) return;
                    const uint32_t sh = (x & sub) << ls;
                    const unsigned c = (atomicAdd(&cnt[x >> s], 1u << sh) >> sh) & cmask;
                    if (g) qb += c;
                    else qa += c;
                });
                each([&](uint32_t x, bool) { cnt[x >> s] = 0u; });
            }
        } else if (est * 48.f < (float)used) {
            walk_lower<false>(row, nlow, deal, &s_grp[1], W, run,
                              [&](const auto& q, const auto& e, const auto& f, auto&) {
                                  each4(q, e, f, [&](uint32_t x, uint32_t) { cnt[x >> s] = 0u; });
                              },
                              norow);
        } else {
            for (int i = tid; i < (used + 3) / 4; i += THREADS) c4[i] = make_uint4(0, 0, 0, 0);
        }
        __syncthreads();
    }
    acc_add(a.ctl, 5, qa + qab);
    acc_add(a.ctl, 11, qb + qab);
    acc_add(a.ctl, 15, wedges);
    acc_add(a.ctl, 20, wedges);
    stage_end(a.ctl, 5);
    stage_end(a.ctl, 9);
}

// A pivot's hash table in shared memory: a slot is an id and a packed count
// (G_a high, G_b low 16 bits; a count is at most the pivot's lower neighbours,
// below 2^15 in every table tier).
constexpr uint32_t TAB_EMPTY = 0xFFFFFFFFu;
struct Table {
    uint32_t *keys, *cnts;
    uint32_t slots;
    __device__ __forceinline__ uint32_t home(uint32_t w) const { return __umulhi(w * 0x9E3779B1u, slots); }
    __device__ __forceinline__ uint32_t next(uint32_t h) const { return h + 1 == slots ? 0u : h + 1; }
    // slots for a pivot of at most wt wedges: 3/4 filled at most
    __device__ static __forceinline__ uint32_t size_for(int wt) { return (uint32_t)(wt + wt / 3 + 32); }
};

// Insert four wedges of pivot u (q[i] null: none); their probes overlap.  Old
// counts are added to qa, qb.
__device__ __forceinline__ void tab_insert(const Table& T, uint32_t u, const uint32_t* const (&q)[PV_UNROLL],
                                           const uint32_t (&e)[PV_UNROLL], const uint32_t (&f)[PV_UNROLL],
                                           unsigned long long& wedges, unsigned long long& qa,
                                           unsigned long long& qb) {
    uint32_t h[PV_UNROLL], inc[PV_UNROLL];
    unsigned todo = 0;
#pragma unroll
    for (int i = 0; i < PV_UNROLL; i++) {
        const uint32_t w = vid(e[i]), both = e[i] & f[i];
        h[i] = T.home(w);
        inc[i] = ((both & FLAG_A) ? 0x10000u : 0u) | (both >> 31);
        if (q[i] && w < u) {
            wedges++;
            if (inc[i]) todo |= 1u << i;
        }
    }
    while (todo) {
        uint32_t k[PV_UNROLL];
#pragma unroll
        for (int i = 0; i < PV_UNROLL; i++) k[i] = (todo >> i) & 1u ? T.keys[h[i]] : 0u;
#pragma unroll
        for (int i = 0; i < PV_UNROLL; i++)
            if (((todo >> i) & 1u) && k[i] == TAB_EMPTY) {
                const uint32_t was = atomicCAS(&T.keys[h[i]], TAB_EMPTY, vid(e[i]));
                k[i] = was == TAB_EMPTY ? vid(e[i]) : was;
            }
#pragma unroll
        for (int i = 0; i < PV_UNROLL; i++)
            if ((todo >> i) & 1u) {
                if (k[i] == vid(e[i])) {
                    const uint32_t c = atomicAdd(&T.cnts[h[i]], inc[i]);
                    if (inc[i] >> 16) qa += c >> 16;
                    if (inc[i] & 1u) qb += c & 0xFFFFu;
                    todo &= ~(1u << i);
                } else {
                    h[i] = T.next(h[i]);
                }
            }
    }
}

// Credits of four wedges (every one was inserted): c_w - 1 to x[i], and to the
// second edge's entry.
template <int MODE>
__device__ __forceinline__ void tab_credit(const Table& T, uint32_t u, const uint32_t* U_col,
                                           unsigned long long* credit, const uint32_t* const (&q)[PV_UNROLL],
                                           const uint32_t (&e)[PV_UNROLL], uint32_t (&x)[PV_UNROLL]) {
#pragma unroll
    for (int i = 0; i < PV_UNROLL; i++) {
        const uint32_t w = vid(e[i]);
        x[i] = 0;
        if (q[i] && w < u) {
            uint32_t h = T.home(w);
            while (T.keys[h] != w) h = T.next(h);
            x[i] = (T.cnts[h] >> 16) - 1;
            if (MODE == C4_EDGE && x[i]) red_u64(&credit[q[i] - U_col], x[i]);
        }
    }
}

// Clear the table; per vertex, every endpoint takes its C(c_w, 2).
template <int MODE>
__device__ __forceinline__ void tab_clear(const Table& T, unsigned long long* credit, uint32_t first, uint32_t step) {
    for (uint32_t i = first; i < T.slots; i += step) {
        if (MODE == C4_VERTEX) {
            const unsigned long long c = T.cnts[i] >> 16;
            if (c >= 2) red_u64(&credit[T.keys[i]], c * (c - 1) / 2);
        }
        T.keys[i] = TAB_EMPTY;
        T.cnts[i] = 0;
    }
}

// Pivots whose endpoints all fit a hash table of SLOTS entries (a bound of at
// most 3/4 SLOTS wedges), a block per pivot.  Only the first 4/3 w~ slots are
// used, so small pivots clear little.
// Measured alone (ncu) on a Chung-Lu graph of 800,000 vertices and 15 M edges:
// 0.65 / 1.27 / 1.06 ms for the small / medium / large table; the kernels
// before (one hash insertion at a time per lane, 32 rows to a warp, the large
// ones in an L2 table) took 10 ms together on the 1.6M/30M graph where these
// take 6.
template <int MODE, int THREADS, int MINB, int SLOTS, int BIN, int WORK>
__global__ void __launch_bounds__(THREADS, MINB) k_c4_table(PivotArgs a, const int32_t* __restrict__ list) {
    pdl_enter();
    extern __shared__ __align__(16) uint32_t sm[];
    constexpr int NW = THREADS / 32;
    uint32_t* const keys = sm;
    uint32_t* const cnts = sm + SLOTS;
    __shared__ C4Task s_task[2];
    __shared__ int s_grp[2];
    const int tid = threadIdx.x, warp = tid >> 5;
    WarpRuns& W = ((WarpRuns*)(sm + 2 * SLOTS))[warp];
    const int npiv = a.ctl->nbin[BIN];
    if (npiv == 0) return;
    for (int i = tid; i < SLOTS; i += THREADS) {
        keys[i] = TAB_EMPTY;
        cnts[i] = 0;
    }
    auto fetch = [&](C4Task& o) {
        o.id = atomicAdd(&a.ctl->work[WORK], 1u);
        if (o.id >= (unsigned)npiv) return;
        o.u = (uint32_t)list[(unsigned)o.id];
        o.rb = a.U_off[o.u];
        o.nlow = a.U_split[o.u];
        o.k = (int)a.U_wt[o.u];
    };
    if (tid == 0) {
        fetch(s_task[0]);
        s_grp[0] = 0;
    }
    unsigned long long qa = 0, qb = 0, wedges = 0;
    __syncthreads();
    for (int it = 0;; it++) {
        const C4Task t = s_task[it & 1];
        if (t.id >= (unsigned)npiv) break;
        const uint32_t u = t.u;
        const uint32_t* const row = a.U_col + t.rb;
        const Table T{keys, cnts, min((uint32_t)SLOTS, Table::size_for(t.k))};
        const Deal deal = deal_groups(t.nlow, (float)t.k, NW);
        auto run = [&](uint32_t fv, const uint32_t** p, int* len) {
            const uint32_t v = vid(fv);
            const long long b = a.U_off[v];
            *p = a.U_col + b;
            *len = (int)(a.U_off[v + 1] - b);
        };
        if (tid == 0) s_grp[1] = 0;
        if (tid == THREADS - 1) fetch(s_task[(it + 1) & 1]);
        unsigned long long old = 0, oldb = 0;
        walk_lower<false>(
            row, t.nlow, deal, &s_grp[0], W, run,
            [&](const auto& q, const auto& e, const auto& f, auto&) {
                tab_insert(T, u, q, e, f, wedges, old, oldb);
            },
            [](unsigned long long, uint32_t, int) {});
        qa += old;
        qb += oldb;
        __syncthreads();
        if (tid == 0) s_grp[0] = 0;
        if (MODE != C4_COUNT) {
            if (MODE == C4_VERTEX) {
                old = warp_sum_u64(old);
                if ((tid & 31) == 0 && old) red_u64(&a.credit[u], old);
            }
            walk_lower<true>(
                row, t.nlow, deal, &s_grp[1], W, run,
                [&](const auto& q, const auto& e, const auto&, auto& x) {
                    tab_credit<MODE>(T, u, a.U_col, a.credit, q, e, x);
                },
                [&](unsigned long long sum, uint32_t fv, int j) {
                    red_u64(&a.credit[MODE == C4_EDGE ? (size_t)(t.rb + j) : (size_t)vid(fv)], sum);
                });
            __syncthreads();
        }
        tab_clear<MODE>(T, a.credit, tid, THREADS);
        __syncthreads();
    }
    acc_add(a.ctl, 5, qa);
    acc_add(a.ctl, 11, qb);
    acc_add(a.ctl, 15, wedges);
    stage_end(a.ctl, 5);
}

// Credits of the small pivots (registers and warp tiers, w~ <= C4_T1): a warp
// per pivot with its own table.
constexpr int CW_WARPS = 8;
constexpr int CW_SLOTS = C4_T1 + C4_T1 / 3 + 32;
struct CreditWarp {
    WarpRuns runs;
    uint32_t keys[CW_SLOTS], cnts[CW_SLOTS];
    int ctr[2];
};
template <int MODE>
__global__ void __launch_bounds__(CW_WARPS * 32, 4) k_c4_warp_credit(PivotArgs a, const int32_t* __restrict__ bins) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char cw_smem[];
    CreditWarp& S = ((CreditWarp*)cw_smem)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int i = lane; i < CW_SLOTS; i += 32) {
        S.keys[i] = TAB_EMPTY;
        S.cnts[i] = 0;
    }
    const int n0 = a.ctl->nbin[BIN_C4_REG], n1 = n0 + a.ctl->nbin[BIN_C4_WARP];
    unsigned long long q = 0, wedges = 0;
    for (int i = gw; i < n1; i += nw) {
        const uint32_t u = (uint32_t)(i < n0 ? bins[(size_t)BIN_C4_REG * a.n + i]
                                             : bins[(size_t)BIN_C4_WARP * a.n + i - n0]);
        const long long rb = a.U_off[u];
        const int nlow = a.U_split[u];
        const Table T{S.keys, S.cnts, min((uint32_t)CW_SLOTS, Table::size_for((int)a.U_wt[u]))};
        const uint32_t* const row = a.U_col + rb;
        const Deal deal{5, 1};  // 32 rows at a time
        auto run = [&](uint32_t fv, const uint32_t** p, int* len) {
            const uint32_t v = vid(fv);
            const long long b = a.U_off[v];
            *p = a.U_col + b;
            *len = (int)(a.U_off[v + 1] - b);
        };
        if (lane < 2) S.ctr[lane] = 0;
        __syncwarp();
        unsigned long long old = 0, oldb = 0;
        walk_lower<false>(
            row, nlow, deal, &S.ctr[0], S.runs, run,
            [&](const auto& qq, const auto& e, const auto& f, auto&) {
                tab_insert(T, u, qq, e, f, wedges, old, oldb);
            },
            [](unsigned long long, uint32_t, int) {});
        __syncwarp();
        q += old;
        if (__any_sync(FULL, old != 0)) {  // else every c_w is 1 at most: no credits
            if (MODE == C4_VERTEX) {
                old = warp_sum_u64(old);
                if (lane == 0) red_u64(&a.credit[u], old);
            }
            walk_lower<true>(
                row, nlow, deal, &S.ctr[1], S.runs, run,
                [&](const auto& qq, const auto& e, const auto&, auto& x) {
                    tab_credit<MODE>(T, u, a.U_col, a.credit, qq, e, x);
                },
                [&](unsigned long long sum, uint32_t fv, int j) {
                    red_u64(&a.credit[MODE == C4_EDGE ? (size_t)(rb + j) : (size_t)vid(fv)], sum);
                });
            __syncwarp();
        }
        tab_clear<MODE>(T, a.credit, lane, 32);
        __syncwarp();
    }
    acc_add(a.ctl, 5, q);
    acc_add(a.ctl, 11, q);
    acc_add(a.ctl, 15, wedges);
    stage_end(a.ctl, 5);
}

// ---- host side -------------------------------------------------------------------

namespace {
constexpr int PV_SMALL = 512, PV_BIG = 1024;
constexpr int PV_BIG_WORDS = 49152;      // 192 KB of counters, one block per SM

template <int SLOTS, int THREADS>
constexpr size_t table_smem() {
    return (size_t)SLOTS * 8 + (size_t)(THREADS / 32) * sizeof(WarpRuns);
}

template <int MODE>
struct C4Kernels {
    static constexpr auto big = k_c4_pivot<MODE, PV_BIG, 1>;
    static constexpr auto small = k_c4_pivot<MODE, PV_SMALL, 2>;
    static constexpr auto tab_s = k_c4_table<MODE, 128, 8, C4_TAB_S, BIN_C4_BSMALL, WORK_C4_BSMALL>;
    static constexpr auto tab_m = k_c4_table<MODE, 512, 2, C4_TAB_M, BIN_C4_BLOCK, WORK_C4_BLOCK>;
    static constexpr auto tab_l = k_c4_table<MODE, 1024, 1, C4_TAB_L, BIN_C4_BIG, WORK_C4_BIG>;

    static void attributes() {
        auto set = [](const void* f, size_t b) {
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b);
        };
        set((const void*)big, (size_t)PV_BIG_WORDS * 4 + (PV_BIG / 32) * sizeof(WarpRuns));
        set((const void*)small, (size_t)(C4_SMALL_IDS / 2 + 128) * 4 + (PV_SMALL / 32) * sizeof(WarpRuns));
        set((const void*)tab_s, table_smem<C4_TAB_S, 128>());
        set((const void*)tab_m, table_smem<C4_TAB_M, 512>());
        set((const void*)tab_l, table_smem<C4_TAB_L, 1024>());
        if constexpr (MODE != C4_COUNT)
            set((const void*)k_c4_warp_credit<MODE>, CW_WARPS * sizeof(CreditWarp));
    }
    static void warps(const PivotArgs& a, const int32_t* bins, int sms, cudaStream_t s) {
        if constexpr (MODE != C4_COUNT)
            k_c4_warp_credit<MODE><<<4 * sms, CW_WARPS * 32, CW_WARPS * sizeof(CreditWarp), s>>>(a, bins);
    }
    static int tables(const PivotArgs& a, const int32_t* bins, int sms, cudaStream_t s, cudaStream_t s2) {
        tab_s<<<8 * sms, 128, table_smem<C4_TAB_S, 128>(), s>>>(a, bins + (size_t)BIN_C4_BSMALL * a.n);
        tab_m<<<2 * sms, 512, table_smem<C4_TAB_M, 512>(), s2>>>(a, bins + (size_t)BIN_C4_BLOCK * a.n);
        tab_l<<<sms, 1024, table_smem<C4_TAB_L, 1024>(), s2>>>(a, bins + (size_t)BIN_C4_BIG * a.n);
        return 3;
    }
    static void pivots(const PivotArgs& a, const C4Geom& g, int c0, cudaStream_t s) {
        if (g.threads == PV_SMALL) small<<<g.ctas, PV_SMALL, g.smem, s>>>(a, c0);
        else big<<<g.ctas, PV_BIG, g.smem, s>>>(a, c0);
    }
};
}  // namespace

C4Geom c4_geom(long long n, int sms) {
    C4Geom g;
    n = std::max<long long>(n, 1);
    g.narrow = n <= 65536;
    const bool small = n <= C4_SMALL_IDS;
    g.threads = small ? PV_SMALL : PV_BIG;
    g.words = small ? (int)((n / 2 + 128) & ~3ll) : PV_BIG_WORDS;
    g.ctas = small ? 3 * sms : sms;
    g.gran = 64;
    while (g.gran < n / 512 && g.gran < 32768) g.gran <<= 1;
    while (g.narrow && (long long)g.gran * PLAN_TILE < n) g.gran <<= 1;  // k_c4_plan: a thread per granule
    g.ngran = (int)((n + g.gran - 1) / g.gran);
    const long long least = (g.narrow ? 2ll * g.words : (long long)g.words) - g.gran + 1;
    g.nchmax = (int)(n / std::max<long long>(least, 1)) + 1 + C4_SPLITS;
    g.group = g.narrow ? g.nchmax : std::min(g.nchmax, 16);
    g.smem = (size_t)g.words * 4 + (size_t)(g.threads / 32) * sizeof(WarpRuns);
    return g;
}

void c4_setup_attributes() {
    C4Kernels<C4_COUNT>::attributes();
    C4Kernels<C4_VERTEX>::attributes();
    C4Kernels<C4_EDGE>::attributes();
}

int enqueue_c4_tables(const PivotArgs& a, int mode, const int32_t* bins, int sms, cudaStream_t s, cudaStream_t s2) {
    return mode == C4_VERTEX ? C4Kernels<C4_VERTEX>::tables(a, bins, sms, s, s2)
           : mode == C4_EDGE ? C4Kernels<C4_EDGE>::tables(a, bins, sms, s, s2)
                             : C4Kernels<C4_COUNT>::tables(a, bins, sms, s, s2);
}

int enqueue_c4_warp_credit(const PivotArgs& a, int mode, const int32_t* bins, int sms, cudaStream_t s) {
    if (mode == C4_VERTEX) C4Kernels<C4_VERTEX>::warps(a, bins, sms, s);
    else C4Kernels<C4_EDGE>::warps(a, bins, sms, s);
    return 1;
}

static int enqueue_c4_runs(const PivotArgs& a, const C4Geom& g, int c0, cudaStream_t s) {
    const int gr = (int)std::max<long long>(
        1, std::min<long long>(((long long)a.n * std::min(g.group, 8) + 255) / 256, 16ll * g.ctas));
    k_c4_runs<<<gr, 256, 0, s>>>(a.U_off, a.U_col, a.n, a.b.head, a.b.chunk, c0, g.group, a.b.run);
    return 1;
}

int enqueue_c4_plan(const PivotArgs& a, const C4Geom& g, cudaStream_t s) {
    int nl = 1;
    if (!g.narrow) {
        k_c4_granules<<<g.ngran, 256, 0, s>>>(a.U_off, a.n, g.gran, a.b.gmax);
        nl++;
    }
    k_c4_plan<<<1, PLAN_TILE, 0, s>>>(a.ctl, a.U_off, a.n, g.gran, g.ngran, g.narrow ? nullptr : a.b.gmax, g.words,
                                      g.ctas, g.nchmax, a.b.head, a.b.chunk);
    return nl + enqueue_c4_runs(a, g, 0, s);
}

int enqueue_c4_pivots(const PivotArgs& a, int mode, const C4Geom& g, cudaStream_t s) {
    int nl = 0;
    for (int c0 = 0; c0 < g.nchmax; c0 += g.group) {
        if (c0) nl += enqueue_c4_runs(a, g, c0, s);
        if (mode == C4_VERTEX) C4Kernels<C4_VERTEX>::pivots(a, g, c0, s);
        else if (mode == C4_EDGE) C4Kernels<C4_EDGE>::pivots(a, g, c0, s);
        else C4Kernels<C4_COUNT>::pivots(a, g, c0, s);
        nl++;
    }
    return nl;
}

}  // namespace gcx
