// gc_region.cu -- the region of change (step a1) and the flagged region
// union graph (step a2).
//
// Region.  W is every vertex within k hops of a batch endpoint (Sec. 4.2:
// a 4-vertex graphlet has diameter at most 3; Algorithm 2 takes the k-hop
// neighbourhood of each changed pair).  The walk starts from all endpoints at
// once, level by level, over a vertex bitmap; each level appends the newly
// reached vertices to the region list, so level L occupies
// wlist[lvl[L-1] .. lvl[L]).  Every inserted or deleted pair joins two
// depth-0 vertices, so walking G alone reaches exactly what walking G u A does.
//
// Union graph.  Row u of U lists N(u) n W plus the insertions A_u, sorted by
// id, each entry tagged FLAG_A / FLAG_B (membership in G_a / G_b).  d_a(u)
// and d_b(u) are the degrees inside G_a and G_b (region-induced, as the
// counts of Algorithm 2 are taken in those graphs), and split(u) is the
// first position whose id exceeds u: the out-list N+(u).
#include "gc_internal.cuh"
#include "gc_kernels.cuh"

namespace gcx {

__device__ __forceinline__ bool in_region(const uint32_t* visited, int32_t v) {
    return (visited[v >> 5] >> (v & 31)) & 1u;
}

// mark v; if it was unmarked, append it to the region list (warp-aggregated)
// (level L, which starts at wlist[first])
__device__ __forceinline__ void visit_append(bool want, int32_t v, uint32_t* visited, int32_t* wlist, int first,
                                             int* count) {
    bool fresh = false;
    if (want) {
        uint32_t bit = 1u << (v & 31);
        if (!(visited[v >> 5] & bit)) fresh = !(atomicOr(&visited[v >> 5], bit) & bit);
    }
    unsigned m = __ballot_sync(FULL, fresh);
    if (m) {
        int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
        int base = 0;
        if (lane == leader) base = first + atomicAdd(count, __popc(m));
        base = __shfl_sync(FULL, base, leader);
        if (fresh) wlist[base + __popc(m & lanemask_lt())] = v;
    }
}

__global__ void k_bfs_sources(Ctl* c, const int32_t* __restrict__ srcA, const int32_t* __restrict__ srcD,
                              uint32_t* __restrict__ visited, int32_t* __restrict__ wlist) {
    pdl_enter();
    stage_begin(c, 1);
    if (c->err) return;
    long long na = c->nA2, nd = c->nD2, tot = na + nd;
    long long stride = (long long)gridDim.x * blockDim.x;
    long long start = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    // the loop bound is warp-uniform so the ballot in visit_append is safe
    long long tot_r = (tot + 31) & ~31ll;
    for (long long i = start; i < tot_r; i += stride) {
        bool ok = i < tot;
        int32_t v = ok ? (i < na ? srcA[i] : srcD[i - na]) : 0;
        visit_append(ok, v, visited, wlist, 0, &c->lcnt[0]);
    }
}

// ends of the levels, for a batch that is committed without a count
__global__ void k_level_ends(Ctl* c) {
    pdl_enter();
    if (threadIdx.x == 0) close_levels(c);
}

// The two-batch form's whole-graph pass: after the batch endpoints (level
// 0), every other vertex joins the region, so W = V and the counts of G_a and
// G_b are those of the whole graph after and before the batch.  An inactive
// batch (a halted run) keeps its empty region.
__global__ void k_region_rest(Ctl* c, int n, uint32_t* __restrict__ visited, int32_t* __restrict__ wlist) {
    pdl_enter();
    if (c->err || !c->active) return;
    const int first = c->lcnt[0];
    const long long n_r = ((long long)n + 31) & ~31ll;  // warp-uniform bound for the ballot
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n_r;
         v += (long long)gridDim.x * blockDim.x)
        visit_append(v < n, (int32_t)(v < n ? v : 0), visited, wlist, first, &c->lcnt[1]);
}

__global__ void k_bfs_expand(Ctl* c, int L, const long long* __restrict__ row_start, const int32_t* __restrict__ deg,
                             const int32_t* __restrict__ col, uint32_t* __restrict__ visited,
                             int32_t* __restrict__ wlist) {
    pdl_enter();
    if (c->err) return;
    int fb = 0, fe = c->lcnt[0];  // the level before
    for (int i = 1; i < L; i++) {
        fb = fe;
        fe += c->lcnt[i];
    }
    int lane = threadIdx.x & 31;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = fb + warp; i < fe; i += nwarps) {
        int32_t x = wlist[i];
        const int32_t* row = col + row_start[x];
        int d = deg[x];
        for (int b = 0; b < d; b += 32) {
            bool ok = b + lane < d;
            int32_t y = ok ? row[b + lane] : 0;
            visit_append(ok, y, visited, wlist, fe, &c->lcnt[L]);
        }
    }
}

// static count: W = V
__global__ void k_region_all(Ctl* c, int n, int32_t* __restrict__ wlist) {
    pdl_enter();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) wlist[i] = i;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->nW = n;
        for (int L = 0; L < MAX_HOPS + 2; L++) {
            c->lvl[L] = n;
            c->lcnt[L] = L == 0 ? n : 0;
        }
    }
}

__global__ void k_u_count(const Ctl* c, const int32_t* __restrict__ wlist, const uint32_t* __restrict__ visited,
                          const long long* __restrict__ row_start, const int32_t* __restrict__ deg,
                          const int32_t* __restrict__ col, const int2* __restrict__ segA,
                          int32_t* __restrict__ U_deg) {
    pdl_enter();
    int nW = c->nW;
    int lane = threadIdx.x & 31;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < nW; i += nwarps) {
        int32_t u = wlist[i];
        const int32_t* row = col + row_start[u];
        int d = deg[u], cnt = 0;
        for (int b = 0; b < d; b += 32) {
            bool ok = b + lane < d && in_region(visited, row[b + lane]);
            cnt += __popc(__ballot_sync(FULL, ok));
        }
        if (lane == 0) {
            int2 a = segA[u];
            U_deg[u] = cnt + (a.y - a.x);
        }
    }
}

__global__ void k_u_fill(const Ctl* c, const int32_t* __restrict__ wlist, const uint32_t* __restrict__ visited,
                         const long long* __restrict__ row_start, const int32_t* __restrict__ deg,
                         const int32_t* __restrict__ col, const int2* __restrict__ segA,
                         const int2* __restrict__ segD, const int32_t* __restrict__ dstA,
                         const int32_t* __restrict__ dstD, const long long* __restrict__ U_off,
                         uint32_t* __restrict__ U_col, int32_t* __restrict__ U_split, int32_t* __restrict__ da,
                         int32_t* __restrict__ db) {
    pdl_enter();
    int nW = c->nW;
    int lane = threadIdx.x & 31;
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < nW; i += nwarps) {
        int32_t u = wlist[i];
        int2 a = segA[u], d = segD[u];
        const int32_t* dl = dstD + d.x;
        long long nd = d.y - d.x, na = a.y - a.x;
        uint32_t* out = U_col + U_off[u];
        long long len = warp_merge_row(
            col + row_start[u], deg[u], dstA + a.x, na, out, FLAG_A,
            [&](int32_t v) { return in_region(visited, v); },
            [&](int32_t v) { return FLAG_B | ((nd == 0 || !sorted_contains(dl, nd, v)) ? FLAG_A : 0u); });
        __syncwarp();
        if (lane == 0) {
            U_split[u] = (int32_t)lower_bound_id(out, len, (uint32_t)u);
            da[u] = (int32_t)(len - nd);
            db[u] = (int32_t)(len - na);
        }
    }
}

// W = V: row u of U is all of N(u) plus the insertions.
__global__ void k_u_count_all(const Ctl* c, const int32_t* __restrict__ wlist, const int32_t* __restrict__ deg,
                              const int2* __restrict__ segA, int32_t* __restrict__ U_deg) {
    pdl_enter();
    const int nW = c->nW;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nW; i += gridDim.x * blockDim.x) {
        const int32_t u = wlist[i];
        U_deg[u] = deg[u] + (segA[u].y - segA[u].x);
    }
}

// Rows of U for W = V.  Every entry is placed by binary searches: a row element
// after the insertions below it, an insertion after the row elements below it.
// TWIN (two independent batches): the kept entries carry the batches' mask in
// their two low bits (dst << 2 | mask, one entry per vertex pair, sorted); a G
// entry loses FLAG_A (FLAG_B) if the first (second) batch deletes it, an
// insertion has FLAG_A (FLAG_B) if the first (second) batch makes it.
//
// Mostly a copy, bound by memory if enough loads are in flight.  A warp per row
// had one row's chain of a dozen dependent loads in flight for 30 entries: 2.66
// ms for the 138 M entries of a 4.8 M-vertex graph, 0.67 now.  So a warp
// takes 32 rows: a lane reads each row's header, and the lanes copy the rows'
// entries as one run, four loads ahead.  Long rows go to the whole block.  The
// rows of a block are spread over the ids in quads, since hubs have
// neighbouring ids.
constexpr int UF_T = 256;
constexpr int U_LONG_ROW = 512;
constexpr int U_LONG_ROWS = 128;  // a block's list of them (a warp copies each further one)
struct UfRow {
    const int32_t* row;
    const int32_t *A, *D;
    uint32_t* out;
    int du, na, nd;
};
template <bool TWIN>
__device__ __forceinline__ void uf_entry(const UfRow& r, int p, int32_t v) {
    uint32_t fl = FLAG_A | FLAG_B;
    const int32_t key = TWIN ? v << 2 : v;
    if (r.nd) {
        const long long q = lower_bound_i32(r.D, r.nd, key);
        if (q < r.nd) {
            const int32_t d = r.D[q];
            if (TWIN ? (d >> 2) == v : d == v)
                fl = TWIN ? fl & ~(((d & 1) ? FLAG_A : 0u) | ((d & 2) ? FLAG_B : 0u)) : FLAG_B;
        }
    }
    r.out[p + (r.na ? lower_bound_i32(r.A, r.na, key) : 0)] = (uint32_t)v | fl;
}
template <bool TWIN>
__device__ __forceinline__ void uf_insertion(const UfRow& r, int q) {
    const int32_t a = r.A[q], x = TWIN ? a >> 2 : a;
    const uint32_t fl = TWIN ? ((a & 1) ? FLAG_A : 0u) | ((a & 2) ? FLAG_B : 0u) : FLAG_A;
    r.out[q + lower_bound_i32(r.row, r.du, x)] = (uint32_t)x | fl;
}
// inclusive prefix sums over the lanes to pre[1 ..], pre[0] = 0; the total
__device__ __forceinline__ int uf_prefix(int x, int* pre) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    pre[lane + 1] = x;
    if (lane == 0) pre[0] = 0;
    __syncwarp();
    return __shfl_sync(FULL, x, 31);
}
template <bool TWIN>
__device__ __forceinline__ void u_fill_rows(const Ctl* c, const int32_t* __restrict__ wlist,
                                            const long long* __restrict__ row_start, const int32_t* __restrict__ deg,
                                            const int32_t* __restrict__ col, const int2* __restrict__ segA,
                                            const int2* __restrict__ segD, const int32_t* __restrict__ dstA,
                                            const int32_t* __restrict__ dstD, const long long* __restrict__ U_off,
                                            uint32_t* __restrict__ U_col, int32_t* __restrict__ U_split,
                                            int32_t* __restrict__ da, int32_t* __restrict__ db) {
    __shared__ UfRow s_row[UF_T], s_long[U_LONG_ROWS];
    __shared__ int s_pre[UF_T / 32][2][33];
    __shared__ int32_t s_longu[U_LONG_ROWS];
    __shared__ int s_nlong, s_cnt[2];
    const int nW = c->nW, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    UfRow* const rows = s_row + 32 * warp;
    int(*const pre)[33] = s_pre[warp];
    if (tid == 0) s_nlong = 0;
    __syncthreads();
    // quad (it, tid / 4) of this block: vertices 4 ((64 it + tid / 4) grid + block) ..
    for (long long it = 0; it * UF_T * gridDim.x + 4ll * blockIdx.x < nW; it++) {
        const long long i = ((it * (UF_T / 4) + (tid >> 2)) * gridDim.x + blockIdx.x) * 4 + (tid & 3);
        UfRow r{};
        int32_t u = 0;
        bool over = false;  // long, and the list is full
        if (i < nW) {
            u = wlist[i];
            const int2 a = segA[u], d = segD[u];
            r.row = col + row_start[u];
            r.A = dstA + a.x;
            r.D = dstD + d.x;
            r.out = U_col + U_off[u];
            r.du = deg[u];
            r.na = a.y - a.x;
            r.nd = d.y - d.x;
            U_split[u] = (int32_t)(lower_bound_i32(r.row, r.du, u + 1) +
                                   (r.na ? lower_bound_i32(r.A, r.na, TWIN ? (u + 1) << 2 : u + 1) : 0));
            if ((long long)r.du + r.na > U_LONG_ROW) {
                const int at = atomicAdd(&s_nlong, 1);
                over = at >= U_LONG_ROWS;
                if (!over) {
                    s_long[at] = r;
                    s_longu[at] = u;
                    r.du = r.na = r.nd = 0;
                    u = -1;
                }
            }
        }
        rows[lane] = r;
        const int total = uf_prefix(over ? 0 : r.du, pre[0]);
        int q = 0;
        for (int b = lane; b < total; b += 128) {
            int at[4], p[4];
            int32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int j = b + 32 * k;
                if (j < total)
                    while (pre[0][q + 1] <= j) q++;
                at[k] = q;
                p[k] = j - pre[0][q];
                v[k] = j < total ? rows[q].row[p[k]] : 0;
            }
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (b + 32 * k < total) uf_entry<TWIN>(rows[at[k]], p[k], v[k]);
        }
        if (__any_sync(FULL, r.na != 0 && !over)) {
            const int ins = uf_prefix(over ? 0 : r.na, pre[1]);
            q = 0;
            for (int j = lane; j < ins; j += 32) {
                while (pre[1][q + 1] <= j) q++;
                uf_insertion<TWIN>(rows[q], j - pre[1][q]);
            }
        }
        for (unsigned m = __ballot_sync(FULL, over); m; m &= m - 1) {
            const UfRow l = rows[__ffs(m) - 1];
            for (int p = lane; p < l.du; p += 32) uf_entry<TWIN>(l, p, l.row[p]);
            for (int p = lane; p < l.na; p += 32) uf_insertion<TWIN>(l, p);
        }
        if (i < nW && u >= 0) {
            int cA = r.na - r.nd, cB = 0;  // insertions into G_a / G_b minus deletions from them
            if (TWIN) {
                cA = 0;
                for (int k = 0; k < r.na; k++) cA += r.A[k] & 1, cB += (r.A[k] >> 1) & 1;
                for (int k = 0; k < r.nd; k++) cA -= r.D[k] & 1, cB -= (r.D[k] >> 1) & 1;
            }
            da[u] = r.du + cA;
            db[u] = r.du + cB;
        }
        __syncwarp();
    }
    __syncthreads();
    for (int k = 0; k < min(s_nlong, U_LONG_ROWS); k++) {
        const UfRow l = s_long[k];
#pragma unroll 4
        for (int p = tid; p < l.du; p += UF_T) uf_entry<TWIN>(l, p, l.row[p]);
        for (int q = tid; q < l.na; q += UF_T) uf_insertion<TWIN>(l, q);
        if (tid < 2) s_cnt[tid] = 0;
        __syncthreads();
        if (TWIN && l.na + l.nd) {
            int cA = 0, cB = 0;
            for (int j = tid; j < l.na; j += UF_T) cA += l.A[j] & 1, cB += (l.A[j] >> 1) & 1;
            for (int j = tid; j < l.nd; j += UF_T) cA -= l.D[j] & 1, cB -= (l.D[j] >> 1) & 1;
            cA = __reduce_add_sync(FULL, cA);
            cB = __reduce_add_sync(FULL, cB);
            if (lane == 0) {
                atomicAdd(&s_cnt[0], cA);
                atomicAdd(&s_cnt[1], cB);
            }
        }
        __syncthreads();
        if (tid == 0) {
            da[s_longu[k]] = l.du + (TWIN ? s_cnt[0] : l.na - l.nd);
            db[s_longu[k]] = l.du + (TWIN ? s_cnt[1] : 0);
        }
        __syncthreads();
    }
}
__global__ void __launch_bounds__(UF_T, 6) k_u_fill_rows(
    const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ row_start,
    const int32_t* __restrict__ deg, const int32_t* __restrict__ col, const int2* __restrict__ segA,
    const int2* __restrict__ segD, const int32_t* __restrict__ dstA, const int32_t* __restrict__ dstD,
    const long long* __restrict__ U_off, uint32_t* __restrict__ U_col, int32_t* __restrict__ U_split,
    int32_t* __restrict__ da, int32_t* __restrict__ db) {
    pdl_enter();
    u_fill_rows<false>(c, wlist, row_start, deg, col, segA, segD, dstA, dstD, U_off, U_col, U_split, da, db);
}
__global__ void __launch_bounds__(UF_T, 6) k_u_fill_twin(
    const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ row_start,
    const int32_t* __restrict__ deg, const int32_t* __restrict__ col, const int2* __restrict__ segA,
    const int2* __restrict__ segD, const int32_t* __restrict__ dstA, const int32_t* __restrict__ dstD,
    const long long* __restrict__ U_off, uint32_t* __restrict__ U_col, int32_t* __restrict__ U_split,
    int32_t* __restrict__ da, int32_t* __restrict__ db) {
    pdl_enter();
    u_fill_rows<true>(c, wlist, row_start, deg, col, segA, segD, dstA, dstD, U_off, U_col, U_split, da, db);
}

// Union rows over the full adjacency (the edge-local path): a block per
// vertex, every entry placed by binary searches (hub rows spread over the
// block).  D entries stay with FLAG_B only, A entries get FLAG_A only.
__global__ void k_u_fill_all(const Ctl* c, const int32_t* __restrict__ wlist, const long long* __restrict__ row_start,
                             const int32_t* __restrict__ deg, const int32_t* __restrict__ col,
                             const int2* __restrict__ segA, const int2* __restrict__ segD,
                             const int32_t* __restrict__ dstA, const int32_t* __restrict__ dstD,
                             const long long* __restrict__ U_off, uint32_t* __restrict__ U_col,
                             int32_t* __restrict__ U_split, int32_t* __restrict__ da, int32_t* __restrict__ db) {
    pdl_enter();
    const int nW = c->nW;
    for (int i = blockIdx.x; i < nW; i += gridDim.x) {
        const int32_t u = wlist[i];
        const int2 a = segA[u], d = segD[u];
        const long long na = a.y - a.x, nd = d.y - d.x;
        const int32_t* row = col + row_start[u];
        const long long len = block_merge_row(row, deg[u], dstA + a.x, na, dstD + d.x, nd, U_col + U_off[u], true,
                                              FLAG_A | FLAG_B, FLAG_A, FLAG_B);
        if (threadIdx.x == 0) {
            U_split[u] = (int32_t)(lower_bound_i32(row, deg[u], u + 1) + lower_bound_i32(dstA + a.x, na, u + 1));
            da[u] = (int32_t)(len - nd);
            db[u] = (int32_t)(len - na);
        }
    }
}

}  // namespace gcx
