// gc_walk.cuh -- walking the rows of a list of neighbours with a block: the
// wedges of a 4-cycle pivot (gc_cycles.cu), the 3-paths of a changed pair
// (gc_local.cu).
#pragma once

#include "gc_internal.cuh"

namespace gcx {

constexpr int PV_UNROLL = 4;

constexpr int PV_LONG = 128;   // a run of at least this many entries is walked by the whole warp

// Per-warp scratch: the short runs of up to 32 lower neighbours.
struct __align__(16) ShortRun {
    const uint32_t* p;
    int len;
    uint32_t fv;
};
struct WarpRuns {
    ShortRun r[32];
};

// How a task's lower neighbours are dealt to warps.  Rows are sorted by id, so
// the last lower neighbours have the longest rows, and those hold most of the
// wedges: groups run from the end of the list, `lev` groups of 2^lm rows, then
// as many of twice the size, and so on up to 32 times the size, so that the
// groups are of similar work and the larger ones come first.  More groups
// balance better, fewer start fewer chains of loads: lev is half a group per
// warp for small tasks and two for large ones.  lm > 0 where runs are shorter
// than 16 entries on average.
struct Deal {
    int lm, lev;
};
__device__ __forceinline__ Deal deal_groups(int nlow, float wedges, int warps) {
    Deal d;
    const int mul = (int)fminf(32.f, 16.f * (float)nlow / fmaxf(wedges, 1.f));
    d.lm = mul >= 1 ? min(5, 32 - __clz(mul)) : 0;
    d.lev = wedges < 512.f * (float)warps ? warps / 2 : wedges < 8192.f * (float)warps ? warps : 2 * warps;
    return d;
}

// Walk up to 32 runs, one per lane: len entries from p, of the neighbour in
// entry fv with index jr (len = 0: none).  Runs of PV_LONG entries and more are
// walked by all lanes, shorter ones by eight lanes a run, four loads in flight
// per lane.  fn(q, e, f, x), which the whole warp calls together, takes four
// entries at a time: q[i] the address (null: none), e[i] the entry, f[i] the
// neighbour's entry; with ACC it returns credits in x[i] (0 where q[i] is null;
// below 2^28, as the lower neighbours of a pivot are), which are summed over
// each run and given to rowfn(sum, fv, jr) by one lane.  (Sums of short runs
// by atomics on their headers, all given at once: eight-lane shuffles at the end
// of each run, which split the warp, took 1.6 ms more of the per-vertex pivots of
// a 1.6M/30M graph.)
template <bool ACC, class Fn, class RowFn>
__device__ __forceinline__ void walk_group(const uint32_t* p, int len, uint32_t fv, int jr, WarpRuns& W, Fn fn,
                                           RowFn rowfn) {
    const int lane = threadIdx.x & 31, sl = lane & 7;
    const bool brief = len > 0 && len < PV_LONG;
    const unsigned ms = __ballot_sync(FULL, brief);
    const int slot = __popc(ms & lanemask_lt());
    const uint32_t* const p0 = p;
    if (brief) W.r[slot] = ShortRun{p, len, fv};
    for (unsigned ml = __ballot_sync(FULL, len >= PV_LONG); ml; ml &= ml - 1) {
        const int src = __ffs(ml) - 1;
        const int n = __shfl_sync(FULL, len, src);
        const uint32_t f0 = __shfl_sync(FULL, fv, src);
        const uint32_t* q0 = (const uint32_t*)__shfl_sync(FULL, (unsigned long long)p, src) + lane;
        unsigned long long acc = 0;
        for (int rem = n - lane; rem + lane > 0; rem -= 32 * PV_UNROLL, q0 += 32 * PV_UNROLL) {
            const uint32_t* q[PV_UNROLL];
            uint32_t e[PV_UNROLL], f[PV_UNROLL], x[PV_UNROLL];
#pragma unroll
            for (int i = 0; i < PV_UNROLL; i++) {
                q[i] = rem > 32 * i ? q0 + 32 * i : nullptr;
                f[i] = f0;
                e[i] = q[i] ? *q[i] : 0u;
            }
            fn(q, e, f, x);
            if (ACC) acc += x[0] + x[1] + x[2] + x[3];
        }
        if (ACC) {
            acc = warp_sum_u64(acc);
            const int js = __shfl_sync(FULL, jr, src);
            if (lane == 0 && acc) rowfn(acc, f0, js);
        }
    }
    __syncwarp();
    const int nr = __popc(ms);
    // eight lanes a run: runs r = lane / 8, + 4, + 8, ...
    int r = (lane >> 3) - 4, rem = 0;
    uint32_t f0 = 0;
    while (__any_sync(FULL, r < nr)) {  // the warp stays together
        const uint32_t* q[PV_UNROLL];
        uint32_t e[PV_UNROLL], f[PV_UNROLL], x[PV_UNROLL];
        int ri[PV_UNROLL];
#pragma unroll
        for (int i = 0; i < PV_UNROLL; i++) {
            r += rem <= 0 ? 4 : 0;
            if (rem <= 0 && r < nr) {
                const ShortRun t = W.r[r];
                p = t.p + sl;
                rem = t.len;
                f0 = t.fv;
            }
            q[i] = rem > sl ? p : nullptr;
            f[i] = f0;
            if (ACC) ri[i] = r;
            p += 8;
            rem -= 8;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < PV_UNROLL; i++) e[i] = q[i] ? *q[i] : 0u;
        fn(q, e, f, x);
        if (ACC) {
            // The eight lanes have read their run's header, so its words take
            // the sums: len the low 16 bits of each credit, p the rest.
            uint32_t acc = 0;
#pragma unroll
            for (int i = 0; i < PV_UNROLL; i++) {
                acc += x[i];
                if (acc && (i + 1 == PV_UNROLL || ri[i + 1] != ri[i])) {
                    ShortRun& t = W.r[ri[i]];
                    atomicAdd((unsigned*)&t.len, acc & 0xFFFFu);
                    if (acc >> 16) atomicAdd((unsigned*)&t.p, acc >> 16);
                    acc = 0;
                }
            }
        }
    }
    __syncwarp();
    if (ACC && brief) {
        const uint32_t lo = *(volatile unsigned*)&W.r[slot].len - (uint32_t)len;
        const uint32_t hi = *(volatile unsigned*)&W.r[slot].p - (uint32_t)(uintptr_t)p0;
        const unsigned long long sum = lo + ((unsigned long long)hi << 16);
        if (sum) rowfn(sum, fv, jr);
    }
    __syncwarp();
}

// Walk the wedges of a pivot with lower neighbours row[0 .. nlow).  run(e, &p,
// &len) gives the entries to walk of the neighbour in entry e.  The warps of
// the block take groups of neighbours from *ctr; each lane looks up one
// neighbour's run (walk_group; its index jr is the one in the row).
template <bool ACC, class RunFn, class Fn, class RowFn>
__device__ __forceinline__ void walk_lower(const uint32_t* __restrict__ row, int nlow, Deal d, int* ctr, WarpRuns& W,
                                           RunFn run, Fn fn, RowFn rowfn) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        int g = 0;
        if (lane == 0) g = atomicAdd(ctr, 1);
        g = __shfl_sync(FULL, g, 0);
        const int q = min(g / d.lev, 5);
        const int gs = (1 << q) << d.lm;
        int j0 = (d.lev * ((1 << q) - 1) << d.lm) + (g - q * d.lev) * gs;
        if (j0 >= nlow) break;
        for (const int je = min(j0 + gs, nlow); j0 < je; j0 += 32) {
            int len = 0, jr = 0;
            const uint32_t* p = nullptr;
            uint32_t fv = 0;
            if (j0 + lane < je) {
                jr = nlow - 1 - j0 - lane;
                fv = row[jr];
                run(fv, &p, &len);
            }
            walk_group<ACC>(p, len, fv, jr, W, fn, rowfn);
        }
    }
}

}  // namespace gcx
