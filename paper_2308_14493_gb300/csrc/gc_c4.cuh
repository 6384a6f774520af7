// gc_c4.cuh -- the 4-cycle pivots counted in shared memory (gc_cycles.cu):
// plan, buffers and launcher, for the counting passes.
#pragma once

#include "gc_internal.cuh"

namespace gcx {

// Add a warp's sum to accumulator `slot`: one atomic per warp, on one of
// ACC_STRIPES copies chosen by the warp (thousands of warps adding to one
// address would queue at a single L2 slice); k_finalize sums the copies.
__device__ __forceinline__ void acc_add_warp(Ctl* c, int slot, unsigned long long x) {
    if ((threadIdx.x & 31) == 0 && x) {
        const int stripe = (int)((blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) & (ACC_STRIPES - 1));
        atomicAdd(&c->accs[slot][stripe], x);
    }
}
__device__ __forceinline__ void acc_add(Ctl* c, int slot, unsigned long long x) {
    acc_add_warp(c, slot, warp_sum_u64(x));
}

// One chunk of ids [lo, hi) whose counters fill the shared array together:
// 32 >> s bits a counter.  share: the chunk's part of all adjacency entries.
struct C4Chunk {
    int lo, hi, s;
    float share;
};
struct C4Head {
    int nch;                    // chunks, highest ids first
    int pad;
    unsigned long long task;    // next (chunk, pivot) of the launch
};

// Up to this many ids, 16-bit counters of all of them take at most 32 KB and
// several blocks share an SM.
constexpr int C4_SMALL_IDS = 16384;

// Launch geometry and buffer sizes of the pivot kernel for ids below n.
struct C4Geom {
    int threads, ctas;          // block size, blocks in all
    int words;                  // 32-bit words of shared counters per block
    int gran, ngran;            // ids per granule (power of two), granules
    bool narrow;                // every degree is below 2^16 (n <= 2^16)
    int nchmax, group;          // bound on the chunks; chunks whose run bounds are held at a time
    size_t smem;
};
C4Geom c4_geom(long long n, int sms);

// Slots of the three hash-table tiers (filled to at most 3/4).
constexpr int C4_TAB_S = 2816, C4_TAB_M = 12288, C4_TAB_L = 26112;

constexpr int C4_LIST = 16384;  // one-graph wedges listed per block
struct C4Bufs {
    C4Head* head;               // 1
    C4Chunk* chunk;             // nchmax
    int32_t* gmax;              // ngran
    unsigned long long* run;    // group * n packed runs (start << 28 | length)
    uint32_t* list;             // ctas * lcap
    long long lcap;
};

// What a walk does with the counts: the global sums only, or credits per
// vertex / per adjacency entry as well.
enum { C4_COUNT = 0, C4_VERTEX = 1, C4_EDGE = 2 };

struct PivotArgs {
    Ctl* ctl;
    const int32_t* pivots;      // BIN_C4_DENSE, by falling wedge bound
    const long long* U_off;
    const uint32_t* U_col;
    const int32_t* U_split;
    const long long* U_wt;
    int n;
    C4Bufs b;
    int words;
    int group;
    unsigned long long* credit;  // C4_VERTEX: per vertex, C4_EDGE: per entry (added to)
};

// Plan and run bounds of the pivots (needs k_wedge_bound's sums; not the bins);
// the hash-table tiers (the small one on stream s, the others on s2) and the
// pivot kernel (bins: the work lists, NBINS * n).  All return the launches made.
int enqueue_c4_plan(const PivotArgs& a, const C4Geom& g, cudaStream_t s);
int enqueue_c4_tables(const PivotArgs& a, int mode, const int32_t* bins, int sms, cudaStream_t s, cudaStream_t s2);
// (the credits of the pivots below the tables: C4_VERTEX and C4_EDGE only)
int enqueue_c4_warp_credit(const PivotArgs& a, int mode, const int32_t* bins, int sms, cudaStream_t s);
int enqueue_c4_pivots(const PivotArgs& a, int mode, const C4Geom& g, cudaStream_t s);
void c4_setup_attributes();

}  // namespace gcx
