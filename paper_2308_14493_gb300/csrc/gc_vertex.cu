// gc_vertex.cu -- per-vertex (local) graphlet counts of the current graph:
// for every vertex v, how many induced connected 4-vertex graphlets hold v
// in each orbit 4..14 (3-path end, middle; 3-star leaf, centre; 4-cycle;
// tailed triangle tail end, other corner, attachment; diamond degree-2,
// degree-3 corner; 4-clique), and their sums per graphlet [g1..g6].
//
// The containment identity behind the global counts (Sec. 3, PGD's closed
// forms) holds per vertex and role: a 4-set S of induced type g holding v
// in orbit o contains a fixed number of copies of each subgraph H with v
// in role r, so the non-induced role counts are N_r(v) = sum_o M[r][o]
// I_o(v), M triangular.  The role counts (d degrees, t_e triangles per
// edge, tri(v) = T2[v] / 2, s(u) = sum_{w in N(u)} (d_w - 1)):
//   3-path   end sum_{u in N(v)} (s(u) - (d_v - 1)) - 2 tri(v);
//            middle sum_{u in N(v)} ((d_v - 1)(d_u - 1) - t_vu)
//   3-star   leaf sum_{u in N(v)} C(d_u - 1, 2); centre C(d_v, 3)
//   4-cycle  counted once at its highest vertex u with opposite corner w:
//            c_w = common lower neighbours, C(c_w, 2) cycles credit u and
//            w, and each middle vertex a of a wedge u-a-w gets c_w - 1
//   tailed triangle  tail end sum_z (tri(z) - t_vz); other corner
//            sum_y t_vy (d_y - 2); attachment tri(v)(d_v - 2)
//   diamond  degree-2 corner: for each triangle {v, a, b}, t_ab - 1;
//            degree-3 corner sum_u C(t_vu, 2)
//   4-clique listed once (oriented), each of its four vertices credited
// The 4-cycle credits come from the counting pass itself (gc_cycles.cu in
// its credit modes, in place of the global 4-cycle kernels), the triangle
// and 4-clique credits from the root kernels below, everything else from one
// row scan at the end.  The input is the union graph U of a static count (both
// flags on every entry, t of each out-entry in tpack, T2 filled, the work bins
// of the triangle roots).
//
// The second half of the file gives the same per edge (ten edge orbits).
#include <algorithm>

#include "gc_internal.cuh"
#include "gc_kernels.cuh"

namespace gcx {

// t of every entry (out-entries carry it; an in-entry reads its twin).
__global__ void k_v_tsym(const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                         const uint32_t* __restrict__ U_col, const int32_t* __restrict__ U_split,
                         const unsigned long long* __restrict__ tpack, uint32_t* __restrict__ tall) {
    pdl_enter();
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < nW; i += nwarps) {
        const uint32_t u = (uint32_t)wlist[i];
        for (long long e = U_off[u] + U_split[u] + lane; e < U_off[u + 1]; e += 32) {
            const uint32_t t = (uint32_t)(tpack[e] >> 32);
            const uint32_t v = vid(U_col[e]);
            tall[e] = t;
            const long long vb = U_off[v];
            tall[vb + lower_bound_id(U_col + vb, U_split[v], u)] = t;
        }
    }
}

// s(u) = sum over the neighbours w of (d_w - 1)
__global__ void k_v_s(const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                      const uint32_t* __restrict__ U_col, long long* __restrict__ sdeg) {
    pdl_enter();
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < nW; i += nwarps) {
        const uint32_t u = (uint32_t)wlist[i];
        long long sum = 0;
        for (long long e = U_off[u] + lane; e < U_off[u + 1]; e += 32) {
            const uint32_t w = vid(U_col[e]);
            sum += U_off[w + 1] - U_off[w] - 1;
        }
        sum = (long long)warp_sum_u64((unsigned long long)sum);
        if (lane == 0) sdeg[u] = sum;
    }
}


// ---- triangles and 4-cliques of a root, credited ------------------------------
//
// As in the counting pass (gc_count.cu): root u, X = the entries of its
// out-list, every entry y of N+(v), v in X, that is also in X closes the
// triangle (u, v, y), listed once.  Here t of every edge is known, so X keeps
// only entries with t > 0 (an edge in no triangle closes none): shorter lists,
// fewer rows to walk.  Credits of a triangle:
//   per vertex  t of the opposite edge - 1 to each corner (diamond degree 2)
//   per edge    degree of the opposite corner - 2 (E_OPP), and the t of the
//               two other edges - 2 (E_OUTER)
// X's adjacency is kept as symmetric bit rows S; the 4-cliques through u and
// X[q] are the triangles of S at q (half of sum over p in S[q] of
// popcount(S[q] & S[p])), those through u, X[q], X[p] popcount(S[q] & S[p]).
// Per edge, the pair credits go to the entry (X[q], X[p]), found by walking the
// candidates a second time, only for roots with a 4-clique.
//
// A lane per out-edge merging two rows in global memory took 187 ms on the
// 1.6M/30M graph (32 lanes on rows of very different lengths, three dependent
// loads a step); the root kernels took 14.6 with a search for every candidate and
// 64-bit sums per triangle in shared memory, and take 9.9.

struct TriCredits {
    unsigned long long* d2;   // per vertex: diamond degree-2 corners
    unsigned long long* k4v;  // per vertex: 4-cliques
    unsigned long long* to;   // per entry, two words: E_OPP, E_OUTER
    unsigned long long* k4e;  // per entry: 4-cliques
};

__device__ __forceinline__ void add_u64(unsigned long long* p, unsigned long long x) {
    if (x) atomicAdd(p, x);
}

__device__ __forceinline__ int find_id(const uint32_t* s, int k, uint32_t y) {
    int lo = 0, hi = k;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s[mid] < y) lo = mid + 1;
        else hi = mid;
    }
    return (lo < k && s[lo] == y) ? lo : -1;
}

// 64-bit sum in two shared words (a 64-bit shared atomic is a loop).
struct Sum64 {
    uint32_t lo, hi;
    __device__ __forceinline__ void add(uint32_t x) {
        if (atomicAdd(&lo, x) > ~x) atomicAdd(&hi, 1u);
    }
    __device__ __forceinline__ unsigned long long get() const { return ((unsigned long long)hi << 32) | lo; }
};

// Shared state of one root with up to KM kept entries.
template <bool EDGE, int KM>
struct RootState {
    long long nb[KM];                 // start of N+(X[q])
    Sum64 t3[EDGE ? KM : 1];          // sum of t of the edges (X[q], X[p]) over its triangles
    uint32_t x[KM];                   // ids
    uint32_t t[KM];                   // t of (u, X[q])
    int pre[KM + 1];                  // candidates before row q
    int at[KM];                       // position in u's out-list
    int dg[EDGE ? KM : 1];            // degrees
    uint32_t bloom[KM];               // a bit per hashed id of X
};

// A candidate that passed the filter: id, its row q, its number.
struct Candidate {
    uint32_t y;
    int q, j;
};

__device__ __forceinline__ uint32_t lt_hash(uint32_t y, int km) { return __umulhi(y * 0x9E3779B1u, 32u * km); }

// The candidates lo .. hi - 1 of a root (rows of X one after the other) by one
// warp: those that a bit filter of X lets pass are queued, and 32 at a time
// searched in X; hit(q, p, slot) for each entry `slot` = (X[q], X[p]).
template <bool EDGE, int KM, class Hit>
__device__ __forceinline__ void walk_candidates(const RootState<EDGE, KM>& S, int k, int lo, int hi,
                                                const uint32_t* __restrict__ U_col, Candidate* queue, Hit hit) {
    const int lane = threadIdx.x & 31;
    int q = 0, end = k, nq = 0;  // q: row of candidate lo
    while (end - q > 1) {
        const int mid = (q + end) >> 1;
        if (S.pre[mid] <= lo) q = mid;
        else end = mid;
    }
    auto drain = [&](int n) {
        if (lane < n) {
            const Candidate c = queue[nq + lane];
            const int p = find_id(S.x, k, c.y);
            if (p >= 0) hit(c.q, p, S.nb[c.q] + (c.j - S.pre[c.q]));
        }
        __syncwarp();
    };
    for (int base = lo; base < hi; base += 128) {
        uint32_t y[4];
        int row[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int j = base + 32 * i + lane;
            if (j < hi)
                while (q + 1 < k && S.pre[q + 1] <= j) q++;
            row[i] = q;
            y[i] = j < hi ? vid(U_col[S.nb[q] + (j - S.pre[q])]) : 0u;
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int j = base + 32 * i + lane;
            const uint32_t h = lt_hash(y[i], KM);
            const bool pass = j < hi && ((S.bloom[h >> 5] >> (h & 31)) & 1u);
            const unsigned m = __ballot_sync(FULL, pass);
            if (pass) queue[nq + __popc(m & lanemask_lt())] = Candidate{y[i], row[i], j};
            nq += __popc(m);
            __syncwarp();
            if (nq >= 32) {
                nq -= 32;
                drain(32);
            }
        }
    }
    const int left = nq;
    nq = 0;
    drain(left);
}

// Credits of one triangle (u, X[q], X[p]) that the bit rows do not give: its
// third edge is entry `slot`.
template <bool EDGE, int KM>
__device__ __forceinline__ void credit_triangle(RootState<EDGE, KM>& S, int q, int p, long long slot, uint32_t t3,
                                                long long du, const TriCredits& cr, unsigned long long& mine) {
    if (EDGE) {
        S.t3[q].add(t3);
        S.t3[p].add(t3);
        add_u64(&cr.to[2 * slot], (unsigned long long)(du - 2));
        add_u64(&cr.to[2 * slot + 1], (unsigned long long)S.t[q] + S.t[p] - 2);
    } else {
        mine += t3 - 1;
    }
}

// Credits of (u, X[q]) or X[q] from its bit row (n: partners p; each(fn) runs
// fn(p) over them): 4-cliques n3, and per vertex t of the opposite edges - 1,
// per edge the opposite corners' degrees - 2 and the outer edges' t - 2.
template <bool EDGE, int KM>
__device__ __forceinline__ void credit_member(const RootState<EDGE, KM>& S, int q, long long rb, uint64_t n,
                                              unsigned long long sum, unsigned long long tsum, uint64_t n3,
                                              const TriCredits& cr) {
    if (EDGE) {
        const long long e = rb + S.at[q];
        add_u64(&cr.to[2 * e], sum - 2 * n);
        add_u64(&cr.to[2 * e + 1], tsum + S.t3[q].get() - 2 * n);
        add_u64(&cr.k4e[e], n3);
    } else {
        add_u64(&cr.d2[S.x[q]], tsum - n);
        add_u64(&cr.k4v[S.x[q]], n3);
    }
}

// Roots with short out-lists: a warp per root.
constexpr int LT_WARPS = 8;
template <bool EDGE>
struct WarpRoot {
    RootState<EDGE, 32> r;
    uint32_t row[32];
    Candidate queue[64];
};
template <bool EDGE>
__global__ void __launch_bounds__(LT_WARPS * 32) k_l_tri_warp(const Ctl* c, const int32_t* __restrict__ list,
                                                              const long long* __restrict__ U_off,
                                                              const uint32_t* __restrict__ U_col,
                                                              const int32_t* __restrict__ U_split,
                                                              const uint32_t* __restrict__ tall, TriCredits cr) {
    pdl_enter();
    __shared__ WarpRoot<EDGE> s_w[LT_WARPS];
    const int lane = threadIdx.x & 31;
    WarpRoot<EDGE>& W = s_w[threadIdx.x >> 5];
    RootState<EDGE, 32>& S = W.r;
    const int cnt = c->nbin[BIN_TRI_WARP];
    for (int i = blockIdx.x * LT_WARPS + (threadIdx.x >> 5); i < cnt; i += gridDim.x * LT_WARPS) {
        const uint32_t u = (uint32_t)list[i];
        const long long ub = U_off[u], ue = U_off[u + 1], rb = ub + U_split[u];
        const int k0 = (int)(ue - rb);
        const uint32_t t = lane < k0 ? tall[rb + lane] : 0u;
        const unsigned keep = __ballot_sync(FULL, t > 0);
        const int k = __popc(keep);
        if (k < 2) continue;
        if (t > 0) {
            const int q = __popc(keep & lanemask_lt());
            S.x[q] = vid(U_col[rb + lane]);
            S.t[q] = t;
            S.at[q] = lane;
        }
        __syncwarp();
        const uint32_t xmax = S.x[k - 1];
        int cq = 0;
        if (lane < k) {
            const uint32_t v = S.x[lane];
            const long long vb = U_off[v], ve = U_off[v + 1], nb = vb + U_split[v];
            S.nb[lane] = nb;
            if (EDGE) S.dg[lane] = (int)(ve - vb);
            cq = (int)lower_bound_id(U_col + nb, ve - nb, xmax + 1);
        }
        int inc = cq;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += y;
        }
        const int total = __shfl_sync(FULL, inc, 31);
        S.pre[lane + 1] = inc;
        if (lane == 0) S.pre[0] = 0;
        W.row[lane] = 0;
        S.bloom[lane] = 0;
        if (EDGE) S.t3[lane] = Sum64{0, 0};
        __syncwarp();
        if (lane < k) {
            const uint32_t h = lt_hash(S.x[lane], 32);
            atomicOr(&S.bloom[h >> 5], 1u << (h & 31));
        }
        __syncwarp();
        unsigned long long mine = 0;
        const long long du = ue - ub;
        walk_candidates(S, k, 0, total, U_col, W.queue, [&](int q, int p, long long slot) {
            atomicOr(&W.row[q], 1u << p);
            atomicOr(&W.row[p], 1u << q);
            credit_triangle<EDGE, 32>(S, q, p, slot, tall[slot], du, cr, mine);
        });
        __syncwarp();
        unsigned n3 = 0;  // 4-cliques through u and X[lane]
        if (lane < k) {
            const uint32_t s = W.row[lane];
            unsigned long long sum = 0, tsum = 0;
            for (uint32_t m = s; m; m &= m - 1) {
                const int p = __ffs(m) - 1;
                n3 += __popc(s & W.row[p]);
                tsum += S.t[p];
                if (EDGE) sum += (unsigned)S.dg[p];
            }
            n3 /= 2;
            credit_member<EDGE, 32>(S, lane, rb, __popc(s), sum, tsum, n3, cr);
        }
        const unsigned any = __ballot_sync(FULL, n3 > 0);
        if (EDGE) {
            if (any)
                walk_candidates(S, k, 0, total, U_col, W.queue, [&](int q, int p, long long slot) {
                    add_u64(&cr.k4e[slot], (unsigned long long)__popc(W.row[q] & W.row[p]));
                });
        } else {
            mine = warp_sum_u64(mine);
            const unsigned all = any ? __reduce_add_sync(FULL, n3) : 0u;
            if (lane == 0) {
                add_u64(&cr.d2[u], mine);
                add_u64(&cr.k4v[u], all / 3);
            }
        }
        __syncwarp();
    }
}

// Roots with longer out-lists: a block per root.
template <bool EDGE, int KM>
struct BlockRoot {
    RootState<EDGE, KM> r;
    uint32_t row[KM * (KM / 32 | 1)];
    Candidate queue[8][64];
};
template <bool EDGE, int KM, int BIN, int WORK>
__global__ void __launch_bounds__(256) k_l_tri_block(Ctl* c, const int32_t* __restrict__ list,
                                                     const long long* __restrict__ U_off,
                                                     const uint32_t* __restrict__ U_col,
                                                     const int32_t* __restrict__ U_split,
                                                     const uint32_t* __restrict__ tall, TriCredits cr) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char lt_smem[];
    BlockRoot<EDGE, KM>& B = *(BlockRoot<EDGE, KM>*)lt_smem;
    RootState<EDGE, KM>& S = B.r;
    __shared__ int s_idx, s_k, s_any;
    __shared__ unsigned long long s_mine, s_all;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = blockDim.x >> 5;
    const int cnt = c->nbin[BIN];
    for (;;) {
        if (tid == 0) {
            s_idx = (int)atomicAdd(&c->work[WORK], 1u);
            s_any = 0;
            s_mine = s_all = 0;
        }
        __syncthreads();
        const int idx = s_idx;
        if (idx >= cnt) break;
        const uint32_t u = (uint32_t)list[idx];
        const long long ub = U_off[u], ue = U_off[u + 1], rb = ub + U_split[u], du = ue - ub;
        if (warp == 0) {
            const int k0 = (int)(ue - rb);
            int k = 0;
            for (int b = 0; b < k0; b += 32) {
                const uint32_t t = b + lane < k0 ? tall[rb + b + lane] : 0u;
                const unsigned keep = __ballot_sync(FULL, t > 0);
                if (t > 0) {
                    const int q = k + __popc(keep & lanemask_lt());
                    S.x[q] = vid(U_col[rb + b + lane]);
                    S.t[q] = t;
                    S.at[q] = b + lane;
                }
                k += __popc(keep);
            }
            if (lane == 0) s_k = k;
        }
        __syncthreads();
        const int k = s_k, W = (k + 31) >> 5, ST = W | 1;  // (odd stride: no bank conflicts)
        if (k < 2) {
            __syncthreads();
            continue;
        }
        const uint32_t xmax = S.x[k - 1];
        for (int q = tid; q < k; q += blockDim.x) {
            const uint32_t v = S.x[q];
            const long long vb = U_off[v], ve = U_off[v + 1], nb = vb + U_split[v];
            S.nb[q] = nb;
            if (EDGE) S.dg[q] = (int)(ve - vb);
            S.pre[q + 1] = (int)lower_bound_id(U_col + nb, ve - nb, xmax + 1);
            if (EDGE) S.t3[q] = Sum64{0, 0};
        }
        for (int j = tid; j < k * ST; j += blockDim.x) B.row[j] = 0;
        for (int j = tid; j < KM; j += blockDim.x) S.bloom[j] = 0;
        __syncthreads();
        for (int q = tid; q < k; q += blockDim.x) {
            const uint32_t h = lt_hash(S.x[q], KM);
            atomicOr(&S.bloom[h >> 5], 1u << (h & 31));
        }
        if (warp == 0) {  // inclusive scan of pre[1..k]
            int carry = 0;
            for (int b = 0; b < k; b += 32) {
                int x = b + lane < k ? S.pre[b + lane + 1] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULL, x, o);
                    if (lane >= o) x += y;
                }
                if (b + lane < k) S.pre[b + lane + 1] = x + carry;
                carry += __shfl_sync(FULL, x, 31);
            }
            if (lane == 0) S.pre[0] = 0;
        }
        __syncthreads();
        const int total = S.pre[k];
        unsigned long long mine = 0;
        const int lo = (int)((long long)total * warp / NW), hi = (int)((long long)total * (warp + 1) / NW);
        walk_candidates(S, k, lo, hi, U_col, B.queue[warp], [&](int q, int p, long long slot) {
            atomicOr(&B.row[q * ST + (p >> 5)], 1u << (p & 31));
            atomicOr(&B.row[p * ST + (q >> 5)], 1u << (q & 31));
            credit_triangle<EDGE, KM>(S, q, p, slot, tall[slot], du, cr, mine);
        });
        __syncthreads();
        unsigned long long all = 0;
        for (int q = tid; q < k; q += blockDim.x) {
            const uint32_t* s = B.row + q * ST;
            unsigned long long n3 = 0, sum = 0, tsum = 0;  // n3: 4-cliques through u and X[q], twice
            unsigned n = 0;
            for (int i = 0; i < W; i++)
                for (uint32_t m = s[i]; m; m &= m - 1) {
                    const int p = i * 32 + __ffs(m) - 1;
                    const uint32_t* r = B.row + p * ST;
                    unsigned x = 0;
                    for (int j = 0; j < W; j++) x += __popc(s[j] & r[j]);
                    n3 += x;
                    tsum += S.t[p];
                    if (EDGE) sum += (unsigned)S.dg[p];
                    n++;
                }
            n3 /= 2;
            all += n3;
            credit_member<EDGE, KM>(S, q, rb, n, sum, tsum, n3, cr);
        }
        if (EDGE) {
            if (all) s_any = 1;
            __syncthreads();
            if (s_any)
                walk_candidates(S, k, lo, hi, U_col, B.queue[warp], [&](int q, int p, long long slot) {
                    unsigned x = 0;
                    for (int j = 0; j < W; j++) x += __popc(B.row[q * ST + j] & B.row[p * ST + j]);
                    add_u64(&cr.k4e[slot], x);
                });
        } else {
            mine = warp_sum_u64(mine);
            all = warp_sum_u64(all);
            if (lane == 0 && (mine | all)) {
                atomicAdd(&s_mine, mine);
                atomicAdd(&s_all, all);
            }
            __syncthreads();
            if (tid == 0) {
                add_u64(&cr.d2[u], s_mine);
                add_u64(&cr.k4v[u], s_all / 3);
            }
        }
        __syncthreads();
    }
}

// Roots with out-lists beyond the block tier: a warp per root, a lane per
// out-edge e = (u, v) merging N+(u) after v with N+(v).
template <bool EDGE>
__global__ void k_l_tri_merge(const Ctl* c, const int32_t* __restrict__ list, const long long* __restrict__ U_off,
                              const uint32_t* __restrict__ U_col, const int32_t* __restrict__ U_split,
                              const uint32_t* __restrict__ tall, TriCredits cr) {
    pdl_enter();
    const int cnt = c->nbin[BIN_TRI_MERGE];
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int wi = warp; wi < cnt; wi += nwarps) {
        const uint32_t u = (uint32_t)list[wi];
        const long long ob = U_off[u] + U_split[u], oe = U_off[u + 1], du = oe - U_off[u];
        for (long long e = ob + lane; e < oe; e += 32) {
            const unsigned long long te = tall[e];
            if (!te) continue;
            const uint32_t v = vid(U_col[e]);
            const long long vb = U_off[v] + U_split[v], ve = U_off[v + 1], dv = ve - U_off[v];
            long long i = e + 1, j = vb;
            unsigned long long k4 = 0;
            while (i < oe && j < ve) {
                const uint32_t x = vid(U_col[i]), y = vid(U_col[j]);
                if (x < y) {
                    i++;
                } else if (x > y) {
                    j++;
                } else {
                    // triangle (u, v, y): t of uv, uy, vy at e, i, j
                    const unsigned long long ti = tall[i], tj = tall[j];
                    const long long yb = U_off[y] + U_split[y], ye = U_off[y + 1], dy = ye - U_off[y];
                    if (EDGE) {
                        add_u64(&cr.to[2 * e], (unsigned long long)(dy - 2));
                        add_u64(&cr.to[2 * e + 1], ti + tj - 2);
                        add_u64(&cr.to[2 * i], (unsigned long long)(dv - 2));
                        add_u64(&cr.to[2 * i + 1], te + tj - 2);
                        add_u64(&cr.to[2 * j], (unsigned long long)(du - 2));
                        add_u64(&cr.to[2 * j + 1], te + ti - 2);
                    } else {
                        add_u64(&cr.d2[u], tj - 1);
                        add_u64(&cr.d2[v], ti - 1);
                        add_u64(&cr.d2[y], te - 1);
                    }
                    // 4-cliques (u, v, y, z), z > y in N+(u), N+(v), N+(y)
                    long long p = i + 1, q = j + 1, r = yb;
                    unsigned long long kk = 0;
                    while (p < oe && q < ve && r < ye) {
                        const uint32_t a = vid(U_col[p]), b = vid(U_col[q]), z = vid(U_col[r]);
                        const uint32_t mx = max(a, max(b, z));
                        if (a == mx && b == mx && z == mx) {
                            if (EDGE) {
                                atomicAdd(&cr.k4e[p], 1ull);
                                atomicAdd(&cr.k4e[q], 1ull);
                                atomicAdd(&cr.k4e[r], 1ull);
                            } else {
                                atomicAdd(&cr.k4v[a], 1ull);
                            }
                            kk++;
                            p++;
                            q++;
                            r++;
                        } else {
                            if (a < mx) p++;
                            if (b < mx) q++;
                            if (z < mx) r++;
                        }
                    }
                    if (EDGE) {
                        add_u64(&cr.k4e[i], kk);
                        add_u64(&cr.k4e[j], kk);
                    } else {
                        add_u64(&cr.k4v[v], kk);
                        add_u64(&cr.k4v[y], kk);
                    }
                    k4 += kk;
                    i++;
                    j++;
                }
            }
            add_u64(EDGE ? &cr.k4e[e] : &cr.k4v[u], k4);
        }
    }
}

template <bool EDGE>
static int enqueue_tri_credits(Ctl* ctl, const int32_t* bins, int n, const long long* U_off, const uint32_t* U_col,
                               const int32_t* U_split, const uint32_t* tall, const TriCredits& cr, int sms,
                               cudaStream_t s, const SideStreams& side) {
    const auto small = k_l_tri_block<EDGE, TRI_KS, BIN_TRI_SMALL, WORK_LT_SMALL>;
    const auto block = k_l_tri_block<EDGE, TRI_KM, BIN_TRI_BLOCK, WORK_LT_BLOCK>;
    constexpr size_t sm_small = sizeof(BlockRoot<EDGE, TRI_KS>), sm_block = sizeof(BlockRoot<EDGE, TRI_KM>);
    cudaFuncSetAttribute(block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_block);
    auto list = [&](int b) { return bins + (size_t)b * n; };
    const cudaStream_t s1 = side.on(1, s), s2 = side.on(2, s);
    if (side.aux[0]) {  // (k_v_tsym, before this on s, has to be done)
        cudaEventRecord(side.fork, s);
        cudaStreamWaitEvent(s1, side.fork, 0);
        cudaStreamWaitEvent(s2, side.fork, 0);
    }
    k_l_tri_warp<EDGE><<<6 * sms, LT_WARPS * 32, 0, s>>>(ctl, list(BIN_TRI_WARP), U_off, U_col, U_split, tall, cr);
    small<<<8 * sms, 256, sm_small, s1>>>(ctl, list(BIN_TRI_SMALL), U_off, U_col, U_split, tall, cr);
    block<<<3 * sms, 256, sm_block, s2>>>(ctl, list(BIN_TRI_BLOCK), U_off, U_col, U_split, tall, cr);
    k_l_tri_merge<EDGE><<<sms, 256, 0, s2>>>(ctl, list(BIN_TRI_MERGE), U_off, U_col, U_split, tall, cr);
    return 4;
}

// ---- per vertex -----------------------------------------------------------------

// The row terms of each vertex, the credits, and the inversion: orbit counts
// by the triangular role containment; out[k v + j] by external id: the eleven
// orbits (k = 11) or their sums per graphlet (k = 6).  A warp per vertex.
__global__ void k_v_finalize(const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                             const uint32_t* __restrict__ U_col, const uint32_t* __restrict__ tall,
                             const long long* __restrict__ sdeg, const unsigned long long* __restrict__ T2,
                             const unsigned long long* __restrict__ d2, const unsigned long long* __restrict__ k4,
                             const unsigned long long* __restrict__ c4, const int32_t* __restrict__ iperm, int k,
                             unsigned long long* __restrict__ out) {
    pdl_enter();
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < nW; i += nwarps) {
        const uint32_t v = (uint32_t)wlist[i];
        const long long rb = U_off[v], re = U_off[v + 1];
        const long long d = re - rb, trv = (long long)(T2[v] / 2);
        long long pe = 0, pm = 0, sl = 0, tl = 0, to = 0, d3 = 0;
        for (long long e = rb + lane; e < re; e += 32) {
            const uint32_t u = vid(U_col[e]);
            const long long du = U_off[u + 1] - U_off[u], t = tall[e];
            pe += sdeg[u] - (d - 1);
            pm += (d - 1) * (du - 1) - t;
            sl += (du - 1) * (du - 2) / 2;
            tl += (long long)(T2[u] / 2) - t;
            to += t * (du - 2);
            d3 += t * (t - 1) / 2;
        }
        pe = (long long)warp_sum_u64((unsigned long long)pe);
        pm = (long long)warp_sum_u64((unsigned long long)pm);
        sl = (long long)warp_sum_u64((unsigned long long)sl);
        tl = (long long)warp_sum_u64((unsigned long long)tl);
        to = (long long)warp_sum_u64((unsigned long long)to);
        d3 = (long long)warp_sum_u64((unsigned long long)d3);
        if (lane == 0) {
            const long long o14 = (long long)k4[v];
            const long long o13 = d3 - 3 * o14;
            const long long o12 = (long long)d2[v] - 3 * o14;
            const long long o11 = trv * (d - 2) - 2 * o13 - 3 * o14;
            const long long o10 = to - 2 * o12 - 2 * o13 - 6 * o14;
            const long long o9 = tl - 2 * o12 - 3 * o14;
            const long long o8 = (long long)c4[v] - o12 - o13 - 3 * o14;
            const long long o7 = d * (d - 1) * (d - 2) / 6 - o11 - o13 - o14;
            const long long o6 = sl - o9 - o10 - 2 * o12 - o13 - 3 * o14;
            const long long o5 = pm - 2 * o8 - o10 - 2 * o11 - 2 * o12 - 4 * o13 - 6 * o14;
            const long long o4 = pe - 2 * trv - 2 * o8 - 2 * o9 - o10 - 4 * o12 - 2 * o13 - 6 * o14;
            unsigned long long* o = out + (size_t)k * iperm[v];
            if (k == 11) {
                const long long orb[11] = {o4, o5, o6, o7, o8, o9, o10, o11, o12, o13, o14};
                for (int j = 0; j < 11; j++) o[j] = (unsigned long long)orb[j];
            } else {
                o[0] = (unsigned long long)(o4 + o5);
                o[1] = (unsigned long long)(o6 + o7);
                o[2] = (unsigned long long)o8;
                o[3] = (unsigned long long)(o9 + o10 + o11);
                o[4] = (unsigned long long)(o12 + o13);
                o[5] = (unsigned long long)o14;
            }
        }
    }
}

// ---------------------------------------------------------------------
// Per-edge (local) counts.  The same containment identity holds per edge
// {u, v} and edge role, with the edge orbits 0..9 (3-path end, middle
// edge; 3-star edge; 4-cycle edge; tailed triangle tail, triangle edge
// opposite the attachment, triangle edge at the attachment; diamond outer
// edge, chord; 4-clique edge).  The non-induced role counts of the edge
// (tri(x) = T2[x] / 2, s(x) = sum_{w in N(x)} (d_w - 1)):
//   3-path end   (s(v) - (d_u - 1) - t) + (s(u) - (d_v - 1) - t)
//   3-path middle (d_u - 1)(d_v - 1) - t;  3-star C(d_u - 1, 2) + C(d_v - 1, 2)
//   4-cycle      credited by the counting pass (gc_cycles.cu)
//   tail         (tri(u) - t) + (tri(v) - t);  attachment t (d_u + d_v - 4)
//   opposite     sum over triangles {u, v, w} of d_w - 2
//   diamond outer  sum over triangles {u, v, w} of t_uw + t_vw - 2
//   chord C(t, 2);  4-clique credited by the clique listing
// 4-cycle credits land on either entry of the edge (the finalize adds both),
// triangle and 4-clique credits on the out-entry.

// One sort key per edge, its external pair (lo << nb) | hi, from the
// out-entries: vertex u's keys start at out_off[u].
__global__ void k_e_outdeg(int n, const long long* __restrict__ U_off, const int32_t* __restrict__ U_split,
                           int32_t* __restrict__ outdeg) {
    pdl_enter();
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x)
        outdeg[u] = (int32_t)(U_off[u + 1] - U_off[u]) - U_split[u];
}
__global__ void k_e_keys(const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                         const uint32_t* __restrict__ U_col, const int32_t* __restrict__ U_split,
                         const int32_t* __restrict__ iperm, int nb, const long long* __restrict__ out_off,
                         unsigned long long* __restrict__ keys) {
    pdl_enter();
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < nW; i += nwarps) {
        const uint32_t u = (uint32_t)wlist[i];
        const long long ob = U_off[u] + U_split[u], to = out_off[u] - ob;
        const unsigned long long a = (unsigned long long)iperm[u];
        for (long long e = ob + lane; e < U_off[u + 1]; e += 32) {
            const unsigned long long b = (unsigned long long)iperm[vid(U_col[e])];
            keys[to + e] = a < b ? (a << nb) | b : (b << nb) | a;
        }
    }
}

// Orbit counts per edge by the triangular edge-role containment.  A warp
// per vertex x, a lane per out-entry e = (x, y); the 4-cycle credits of the
// twin entry (x in y's row) are added, the edge's row in the output is the rank
// of its key among the sorted keys.  out[k row + j]: the ten edge orbits
// (k = 10) or their sums per graphlet (k = 6); edges[2 row] = (lo, hi).
__global__ void k_e_finalize(const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ U_off,
                             const uint32_t* __restrict__ U_col, const int32_t* __restrict__ U_split,
                             const uint32_t* __restrict__ tall, const long long* __restrict__ sdeg,
                             const unsigned long long* __restrict__ T2, const unsigned long long* __restrict__ to,
                             const unsigned long long* __restrict__ k4, const unsigned long long* __restrict__ c4,
                             const int32_t* __restrict__ iperm, const unsigned long long* __restrict__ skeys,
                             int nb, long long m, int k, unsigned long long* __restrict__ out,
                             int32_t* __restrict__ edges) {
    pdl_enter();
    const int nW = c->nW;
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < nW; i += nwarps) {
        const uint32_t x = (uint32_t)wlist[i];
        const long long dx = U_off[x + 1] - U_off[x], trx = (long long)(T2[x] / 2), sx = sdeg[x];
        const unsigned long long ex = (unsigned long long)iperm[x];
        for (long long e = U_off[x] + U_split[x] + lane; e < U_off[x + 1]; e += 32) {
            const uint32_t y = vid(U_col[e]);
            const long long yb = U_off[y];
            const long long tw = yb + lower_bound_id(U_col + yb, U_split[y], x);
            const long long dy = U_off[y + 1] - yb, t = tall[e];
            const long long n_opp = (long long)to[2 * e], n_outer = (long long)to[2 * e + 1];
            const long long n_c4 = (long long)(c4[e] + c4[tw]), n_k4 = (long long)k4[e];
            const long long n_pend = (sdeg[y] - (dx - 1) - t) + (sx - (dy - 1) - t);
            const long long n_pmid = (dx - 1) * (dy - 1) - t;
            const long long n_star = (dx - 1) * (dx - 2) / 2 + (dy - 1) * (dy - 2) / 2;
            const long long n_tail = (trx - t) + ((long long)(T2[y] / 2) - t);
            const long long n_att = t * (dx + dy - 4);
            const long long n_chord = t * (t - 1) / 2;
            const long long i9 = n_k4;
            const long long i8 = n_chord - i9;
            const long long i7 = n_outer - 4 * i9;
            const long long i6 = n_att - 4 * i8 - i7 - 4 * i9;
            const long long i5 = n_opp - i7 - 2 * i9;
            const long long i4 = n_tail - i7 - 2 * i9;
            const long long i3 = n_c4 - i7 - 2 * i9;
            const long long i2 = n_star - i6 - i4 - 2 * i8 - i7 - 2 * i9;
            const long long i1 = n_pmid - i3 - i6 - 2 * i8 - i7 - 2 * i9;
            const long long i0 = n_pend - 2 * i3 - 2 * i5 - 2 * i4 - 3 * i7 - 4 * i9;
            // rank of the key among the m sorted edge keys
            const unsigned long long ey = (unsigned long long)iperm[y];
            const unsigned long long lo = ex < ey ? ex : ey, hi = ex < ey ? ey : ex;
            const unsigned long long key = (lo << nb) | hi;
            long long a = 0, b = m;
            while (a < b) {
                const long long mid = (a + b) >> 1;
                if (skeys[mid] < key) a = mid + 1;
                else b = mid;
            }
            unsigned long long* o = out + (size_t)k * a;
            if (k == 10) {
                o[0] = (unsigned long long)i0; o[1] = (unsigned long long)i1; o[2] = (unsigned long long)i2;
                o[3] = (unsigned long long)i3; o[4] = (unsigned long long)i4; o[5] = (unsigned long long)i5;
                o[6] = (unsigned long long)i6; o[7] = (unsigned long long)i7; o[8] = (unsigned long long)i8;
                o[9] = (unsigned long long)i9;
            } else {
                o[0] = (unsigned long long)(i0 + i1);
                o[1] = (unsigned long long)i2;
                o[2] = (unsigned long long)i3;
                o[3] = (unsigned long long)(i4 + i5 + i6);
                o[4] = (unsigned long long)(i7 + i8);
                o[5] = (unsigned long long)i9;
            }
            if (edges) {
                edges[2 * a] = (int32_t)lo;
                edges[2 * a + 1] = (int32_t)hi;
            }
        }
    }
}

int enqueue_edge_counts(const EdgeArgs& a, cudaStream_t s) {
    const int gw = 8 * a.sms, tpb = 256;
    int nl = 0;
    // the order of the result rows (keys and their sort) beside the credits, and
    // their three tiers beside each other: 655 -> 602 us on 7,000 vertices
    // and 100,000 edges
    a.side.begin(s);
    const cudaStream_t s0 = a.side.on(0, s);
    k_v_s<<<gw, tpb, 0, s0>>>(a.ctl, a.wlist, a.U_off, a.U_col, a.sdeg);
    pdl_launch(k_e_outdeg, dim3(std::max(1, std::min(gw, (a.n + 255) / 256))), dim3(256), 0, s0, a.n, a.U_off,
               a.U_split, a.outdeg);
    nl += 2;
    nl += scan_i32_to_i64(a.outdeg, a.out_off, nullptr, a.n, a.bsum, scan_grid(a.n, a.sms), nullptr, s0);
    pdl_launch(k_e_keys, dim3(gw), dim3(tpb), 0, s0, a.ctl, a.wlist, a.U_off, a.U_col, a.U_split, a.iperm, a.nb,
               a.out_off, a.keys);
    nl++;
    nl += radix_sort_u64((uint64_t*)a.keys, (uint64_t*)a.keys_tmp, a.out_off + a.n, a.m, 2 * a.nb, a.hist, a.sort_grid,
                         s0);
    k_v_tsym<<<gw, tpb, 0, s>>>(a.ctl, a.wlist, a.U_off, a.U_col, a.U_split, a.tpack, a.tall);
    nl++;
    const TriCredits cr{nullptr, nullptr, a.to, a.k4};
    nl += enqueue_tri_credits<true>(a.ctl, a.bins, a.n, a.U_off, a.U_col, a.U_split, a.tall, cr, a.sms, s, a.side);
    a.side.end(s);
    k_e_finalize<<<gw, tpb, 0, s>>>(a.ctl, a.wlist, a.U_off, a.U_col, a.U_split, a.tall, a.sdeg,
               a.T2, a.to, a.k4, a.c4, a.iperm, a.keys, a.nb, a.m, a.orbits ? 10 : 6, a.out, a.edges);
    nl++;
    return nl;
}

int enqueue_vertex_counts(const VertexArgs& a, cudaStream_t s) {
    const int gw = 8 * a.sms, tpb = 256;
    int nl = 0;
    a.side.begin(s);
    k_v_s<<<gw, tpb, 0, a.side.on(0, s)>>>(a.ctl, a.wlist, a.U_off, a.U_col, a.sdeg);
    k_v_tsym<<<gw, tpb, 0, s>>>(a.ctl, a.wlist, a.U_off, a.U_col, a.U_split, a.tpack, a.tall);
    const TriCredits cr{a.d2, a.k4, nullptr, nullptr};
    nl += enqueue_tri_credits<false>(a.ctl, a.bins, a.n, a.U_off, a.U_col, a.U_split, a.tall, cr, a.sms, s, a.side);
    a.side.end(s);
    k_v_finalize<<<gw, tpb, 0, s>>>(a.ctl, a.wlist, a.U_off, a.U_col, a.tall, a.sdeg, a.T2, a.d2,
               a.k4, a.c4, a.iperm, a.orbits ? 11 : 6, a.out);
    nl += 3;
    return nl;
}

}  // namespace gcx
