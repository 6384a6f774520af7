// gc_sort.cu -- device-wide primitives with device-resident lengths:
// LSD radix sort of uint64 keys and exclusive prefix sums.
//
// Both use a fixed grid whose blocks each own one contiguous chunk of the
// input, so the chunk bounds depend only on the length read on the device.
// That keeps every launch shape independent of the data, which lets a whole
// batch pipeline be captured once in a CUDA graph and replayed for batches of
// any size up to the planned maximum.
#include "gc_internal.cuh"

namespace gcx {

namespace {

constexpr int RS_BLOCK = 256;  // threads per block = number of 8-bit digits
constexpr int RS_WARPS = RS_BLOCK / 32;

__device__ __forceinline__ void chunk_of(long long n, long long& beg, long long& end) {
    long long G = gridDim.x;
    long long chunk = (n + G - 1) / G;
    beg = (long long)blockIdx.x * chunk;
    end = beg + chunk < n ? beg + chunk : n;
    if (beg > n) beg = n;
}

__global__ void __launch_bounds__(RS_BLOCK) k_rs_hist(const uint64_t* __restrict__ keys, const long long* d_count,
                                                     int shift, uint32_t* __restrict__ hist) {
    pdl_enter();
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    long long beg, end;
    chunk_of(*d_count, beg, end);
    for (long long i = beg + threadIdx.x; i < end; i += RS_BLOCK) atomicAdd(&h[(keys[i] >> shift) & 255], 1u);
    __syncthreads();
    hist[(size_t)blockIdx.x * 256 + threadIdx.x] = h[threadIdx.x];
}

// Where this block's keys of each digit go: the keys of smaller digits in all
// blocks, then those of the digit in earlier blocks.  hist holds a row of 256
// counts per block; thread d sums column d (coalesced across the block), so no
// scan kernel stands between the histogram and the scatter (one block scanning
// 256 x 304 counts took 107 us a pass; reading them costs each block a few us).
__device__ __forceinline__ uint32_t digit_base(const uint32_t* __restrict__ hist) {
    __shared__ uint32_t wsum[RS_WARPS];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, me = blockIdx.x, G = gridDim.x;
    uint32_t before = 0, all = 0;
#pragma unroll 8
    for (int b = 0; b < G; b++) {
        const uint32_t x = hist[(size_t)b * 256 + t];
        all += x;
        before += b < me ? x : 0u;
    }
    uint32_t y = all;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t z = __shfl_up_sync(FULL, y, o);
        if (lane >= o) y += z;
    }
    if (lane == 31) wsum[warp] = y;
    __syncthreads();
    uint32_t w = 0;
    for (int k = 0; k < warp; k++) w += wsum[k];
    return w + y - all + before;
}

// Stable scatter: each tile of RS_BLOCK keys is ranked within warps with
// __match_any_sync, warp counts are scanned per digit, and a running
// per-digit base carries the order across tiles.
__global__ void __launch_bounds__(RS_BLOCK) k_rs_scatter(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                        const long long* d_count, int shift,
                                                        const uint32_t* __restrict__ hist) {
    pdl_enter();
    __shared__ uint32_t base[256];
    __shared__ uint32_t wcnt[RS_WARPS][256];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    base[t] = digit_base(hist);
    long long beg, end;
    chunk_of(*d_count, beg, end);
    for (long long tile = beg; tile < end; tile += RS_BLOCK) {
#pragma unroll
        for (int w = 0; w < RS_WARPS; w++) wcnt[w][t] = 0;
        __syncthreads();
        long long i = tile + t;
        bool valid = i < end;
        uint64_t key = valid ? in[i] : 0;
        unsigned d = valid ? (unsigned)((key >> shift) & 255) : 256u + (unsigned)lane;
        unsigned peers = __match_any_sync(FULL, d);
        unsigned rank = __popc(peers & lanemask_lt());
        if (valid && lane == __ffs(peers) - 1) wcnt[warp][d] = __popc(peers);
        __syncthreads();
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; w++) {
            uint32_t c = wcnt[w][t];
            wcnt[w][t] = run;
            run += c;
        }
        __syncthreads();
        if (valid) out[base[d] + wcnt[warp][d] + rank] = key;
        __syncthreads();
        base[t] += run;
    }
}

__global__ void k_copy_u64(const uint64_t* __restrict__ in, uint64_t* __restrict__ out, const long long* d_count) {
    pdl_enter();
    long long n = *d_count;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = in[i];
}

// ---- scan -----------------------------------------------------------------

constexpr int SC_BLOCK = 512;

__device__ __forceinline__ long long block_incl_scan_i64(long long x, long long* sh) {
    // sh: at least 32 entries
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        long long w = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w;
    }
    __syncthreads();
    long long r = x + (warp > 0 ? sh[warp - 1] : 0);
    __syncthreads();
    return r;
}

// One or two scans of the same length in a launch (blockIdx.y picks one).
struct ScanJob {
    const int32_t* in;
    long long* out;
    long long* total;
};
constexpr int SC_SUMS = 1024;  // bsum words per scan

// a block's part of the entries, from a multiple of four
__device__ __forceinline__ void scan_chunk(long long n, long long& beg, long long& end) {
    const long long chunk = ((n + gridDim.x - 1) / gridDim.x + 3) & ~3ll;
    beg = min(n, (long long)blockIdx.x * chunk);
    end = min(n, beg + chunk);
}

__global__ void __launch_bounds__(SC_BLOCK) k_scan_partials(ScanJob j0, ScanJob j1, const long long* d_len,
                                                           long long host_len, long long* __restrict__ bsum) {
    pdl_enter();
    __shared__ long long sh[32];
    const int32_t* __restrict__ in = (blockIdx.y ? j1 : j0).in;
    long long n = d_len ? *d_len : host_len;
    long long beg, end;
    scan_chunk(n, beg, end);
    long long s = 0;
#pragma unroll 4
    for (long long i = beg + threadIdx.x; i < end; i += SC_BLOCK) s += in[i];
    s = block_incl_scan_i64(s, sh);
    if (threadIdx.x == SC_BLOCK - 1) bsum[SC_SUMS * blockIdx.y + blockIdx.x] = s;
}

// Four entries a thread and tile: the tiles of a block are a chain of five
// barriers each (10,000 pairs on 7,000 vertices: normalisation 60 -> 50 us,
// with two scans in one launch).
__global__ void __launch_bounds__(SC_BLOCK) k_scan_apply(ScanJob j0, ScanJob j1, const long long* d_len,
                                                        long long host_len, const long long* __restrict__ bsum) {
    pdl_enter();
    __shared__ long long sh[32];
    const ScanJob j = blockIdx.y ? j1 : j0;
    const int32_t* __restrict__ in = j.in;
    long long* __restrict__ out = j.out;
    bsum += SC_SUMS * blockIdx.y;
    long long n = d_len ? *d_len : host_len;
    long long beg, end;
    scan_chunk(n, beg, end);
    // the chunks before this one (at most 1,024 sums: two loads a thread, in
    // place of a kernel that scans them)
    __shared__ long long s_run;
    long long before = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += SC_BLOCK) before += bsum[b];
    before = block_incl_scan_i64(before, sh);
    if (threadIdx.x == SC_BLOCK - 1) s_run = before;
    __syncthreads();
    long long run = s_run;
    const bool wide = (((uintptr_t)in | (uintptr_t)out) & 15) == 0;
    for (long long tile = beg; tile < end; tile += 4 * SC_BLOCK) {
        const long long i = tile + 4 * threadIdx.x;
        int4 x = make_int4(0, 0, 0, 0);
        if (wide && i + 3 < end) {
            x = *(const int4*)(in + i);
        } else {
            if (i < end) x.x = in[i];
            if (i + 1 < end) x.y = in[i + 1];
            if (i + 2 < end) x.z = in[i + 2];
            if (i + 3 < end) x.w = in[i + 3];
        }
        const long long mine = (long long)x.x + x.y + x.z + x.w;
        const long long inc = block_incl_scan_i64(mine, sh);
        const long long o0 = run + inc - mine, o1 = o0 + x.x, o2 = o1 + x.y, o3 = o2 + x.z;
        if (wide && i + 3 < end) {
            *(longlong2*)(out + i) = make_longlong2(o0, o1);
            *(longlong2*)(out + i + 2) = make_longlong2(o2, o3);
        } else {
            if (i < end) out[i] = o0;
            if (i + 1 < end) out[i + 1] = o1;
            if (i + 2 < end) out[i + 2] = o2;
            if (i + 3 < end) out[i + 3] = o3;
        }
        // total of this tile = inclusive value of the last thread
        __shared__ long long tile_total;
        if (threadIdx.x == SC_BLOCK - 1) tile_total = inc;
        __syncthreads();
        run += tile_total;
        __syncthreads();
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        // (with chunks of whole fours the last blocks may be empty; their run
        // is the total all the same)
        out[n] = run;
        if (j.total) *j.total = run;
    }
}

}  // namespace

// One block per 1024 keys (four tiles: short serial scatter loops for the
// small sorts of a batch), at most two per SM.
int radix_grid(long long max_count, int sms) {
    long long g = (max_count + 1023) / 1024;
    if (g < 1) g = 1;
    if (g > 2L * sms) g = 2L * sms;
    if (g > 1024) g = 1024;
    return (int)g;
}

int radix_sort_u64(uint64_t* keys, uint64_t* tmp, const long long* d_count, long long max_count, int bits,
                   uint32_t* hist, int grid, cudaStream_t s) {
    int passes = (bits + 7) / 8;
    int launches = 2 * passes;
    uint64_t* a = keys;
    uint64_t* b = tmp;
    for (int p = 0; p < passes; p++) {
        int shift = 8 * p;
        pdl_launch(k_rs_hist, dim3(grid), dim3(RS_BLOCK), 0, s, a, d_count, shift, hist);
        pdl_launch(k_rs_scatter, dim3(grid), dim3(RS_BLOCK), 0, s, a, b, d_count, shift, hist);
        uint64_t* t = a;
        a = b;
        b = t;
    }
    if (a != keys) {
        int g = (int)((max_count + 255) / 256);
        if (g < 1) g = 1;
        if (g > 2048) g = 2048;
        pdl_launch(k_copy_u64, dim3(g), dim3(256), 0, s, a, keys, d_count);
        launches++;
    }
    return launches;
}

int scan_grid(long long max_len, int sms) {
    long long g = (max_len + 8191) / 8192;
    if (g < 1) g = 1;
    if (g > 4L * sms) g = 4L * sms;
    if (g > 1024) g = 1024;
    return (int)g;
}

static int scan_jobs(const ScanJob& a, const ScanJob& b, int jobs, const long long* d_len, long long host_len,
                     long long* bsum, int grid, cudaStream_t s) {
    pdl_launch(k_scan_partials, dim3(grid, jobs), dim3(SC_BLOCK), 0, s, a, b, d_len, host_len, bsum);
    pdl_launch(k_scan_apply, dim3(grid, jobs), dim3(SC_BLOCK), 0, s, a, b, d_len, host_len, bsum);
    return 2;
}

int scan_i32_to_i64(const int32_t* in, long long* out, const long long* d_len, long long host_len, long long* bsum,
                    int grid, long long* total_out, cudaStream_t s) {
    const ScanJob j{in, out, total_out};
    return scan_jobs(j, j, 1, d_len, host_len, bsum, grid, s);
}

int scan2_i32_to_i64(const int32_t* in0, long long* out0, long long* total0, const int32_t* in1, long long* out1,
                     long long* total1, const long long* d_len, long long* bsum, int grid, cudaStream_t s) {
    return scan_jobs(ScanJob{in0, out0, total0}, ScanJob{in1, out1, total1}, 2, d_len, 0, bsum, grid, s);
}

}  // namespace gcx
