// Values of S into the order of S^T through shared memory.
//
// A pass over S^T reads the values in S^T order; the caller keeps them in S
// order.  Fetching them one by one (permute_kernel in fmm_plan.cu) costs a
// 32-byte sector per 4-byte value.  Here both sides are cut into tiles of W
// values and every value moves twice, each time inside shared memory:
//   pass 1, a block per tile of S: reads its values in order, puts each at its
//     place in shared memory, grouped by the S^T tile it belongs to, and writes
//     every group as one run into the staging array, which lists for each S^T
//     tile the runs of all S tiles;
//   pass 2, a block per tile of S^T: reads its part of the staging array in
//     order, puts each value at its slot in shared memory and writes the tile
//     in order.
// Every access to global memory is a contiguous run, so what bounds it is HBM:
// 4 + 2 + 4 bytes per value and pass (value, 16-bit place, value), 20 in all,
// beside 12 for the single gather, which moves 40.  Pass 1 pays for runs that
// start and end inside a 32-byte sector, so W is the largest that fits: a run
// of a pattern without structure holds W^2 / nnz values (30 at 80M).  Measured
// on GB300, W = 49152: 79.6M values of Zipf rows 358 us (pass 1 208, pass 2 145;
// W = 24576: 390 + 142), 33.6M of Erdos-Renyi rows 148, 19.9M 86; the
// permutation in windows of 2^23 slots (a scatter into L2-sized windows, then a
// gather inside each), which stays for more than 2^28 values, took 547, 237 and
// 139.
//
// A warp of pass 1 writes 32 consecutive values of shared memory: a bit per
// value marks the first of a run, a count per 32 values the runs before them,
// and the run's number gives the distance to its place in the staging array
// (0.2 bytes per value).  Places, marks and distances are built once per plan.
// The order of a run's values in the staging array is whatever the build's counters gave;
// pass 2 undoes it, so the result is exactly vals_t[q] = vals[perm[q]].
#include <algorithm>
#include <atomic>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

__global__ void inverse_kernel(const int32_t *perm, int64_t nnz, uint32_t *inv)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += stride)
        inv[perm[q]] = (uint32_t)q;
}

// run[t][b] = values of S tile t that belong to S^T tile b.
__global__ void __launch_bounds__(512) run_count_kernel(const uint32_t *inv, int64_t nnz, int W,
                                                        int tiles, int32_t *run)
{
    extern __shared__ int32_t cnt[];
    const int64_t base = (int64_t)blockIdx.x * W;
    const int n = (int)min((int64_t)W, nnz - base);
    for (int b = threadIdx.x; b < tiles; b += blockDim.x) cnt[b] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&cnt[inv[base + i] / W], 1);
    __syncthreads();
    for (int b = threadIdx.x; b < tiles; b += blockDim.x)
        run[(size_t)blockIdx.x * tiles + b] = cnt[b];
}

// run[t][b] := place of the run in the staging array (the exclusive sum over
// the S tiles before t, from the start of S^T tile b).
__global__ void run_place_kernel(int W, int tiles, int32_t *run)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= tiles)
        return;
    int64_t at = (int64_t)b * W;
#pragma unroll 8
    for (int t = 0; t < tiles; ++t) {
        const int32_t c = run[(size_t)t * tiles + b];
        run[(size_t)t * tiles + b] = (int32_t)at;
        at += c;
    }
}

// Tables of one S tile: pos1 of every value in shared memory (runs in the
// order of their S^T tile), pos2 of every staged value in its S^T tile, and
// the runs that have values: a bit at the first value of each, for every 32
// values the runs that start before them, and dist = staging place - place in
// shared memory by run number, in place of the tile's row of run.
constexpr int kBuildThreads = 512;
constexpr int kRunsPerThread = 11;   // tiles <= kTilesMax = 512 x 11
__global__ void __launch_bounds__(kBuildThreads)
    tile_places_kernel(const uint32_t *inv, int64_t nnz, int W, int tiles, int32_t *run,
                       uint16_t *pos1, uint16_t *pos2, uint32_t *first, uint16_t *before)
{
    extern __shared__ int32_t cnt[];   // tiles counts, then next places
    __shared__ int32_t part[kBuildThreads], runs[kBuildThreads];
    __shared__ uint32_t mark[kTileValuesMax / 32];
    const int tid = threadIdx.x;
    const int64_t base = (int64_t)blockIdx.x * W;
    const int n = (int)min((int64_t)W, nnz - base), words = W / 32;
    for (int b = tid; b < tiles; b += kBuildThreads) cnt[b] = 0;
    for (int w = tid; w < words; w += kBuildThreads) mark[w] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += kBuildThreads) atomicAdd(&cnt[inv[base + i] / W], 1);
    __syncthreads();
    // exclusive sums of the counts and of the runs: a contiguous piece of the
    // tiles per thread
    const int per = (tiles + kBuildThreads - 1) / kBuildThreads;
    const int b0 = min(tiles, tid * per), b1 = min(tiles, b0 + per);
    int sum = 0, nr = 0;
    for (int b = b0; b < b1; ++b) { sum += cnt[b]; nr += cnt[b] > 0; }
    part[tid] = sum; runs[tid] = nr;
    __syncthreads();
    for (int off = 1; off < kBuildThreads; off <<= 1) {
        const int v = tid >= off ? part[tid - off] : 0, u = tid >= off ? runs[tid - off] : 0;
        __syncthreads();
        part[tid] += v; runs[tid] += u;
        __syncthreads();
    }
    int at = part[tid] - sum;
    int32_t *rn = run + (size_t)blockIdx.x * tiles;
    int32_t dist[kRunsPerThread];
#pragma unroll
    for (int k = 0; k < kRunsPerThread; ++k) {
        const int b = b0 + k;
        dist[k] = 0;
        if (b >= b1)
            continue;
        const int c = cnt[b];
        dist[k] = rn[b] - at;
        rn[b] = dist[k];   // read below by the whole block
        cnt[b] = at;
        if (c > 0)
            atomicOr(&mark[at / 32], 1u << (at % 32));
        at += c;
    }
    __syncthreads();
    for (int i = tid; i < n; i += kBuildThreads) {
        const uint32_t q = inv[base + i];
        const int b = (int)(q / W);
        const int lp = atomicAdd(&cnt[b], 1);
        pos1[base + i] = (uint16_t)lp;
        pos2[(int64_t)rn[b] + lp] = (uint16_t)(q - (uint32_t)b * W);
    }
    __syncthreads();
    // the row of run by run number
    int o = runs[tid] - nr;
    int begin = part[tid] - sum;
#pragma unroll
    for (int k = 0; k < kRunsPerThread; ++k) {
        const int b = b0 + k;
        if (b >= b1)
            continue;
        const int end = cnt[b];   // the place after the run's last value
        if (end > begin)
            rn[o++] = dist[k];
        begin = end;
    }
    // runs that start before each 32 values: a contiguous piece of the words
    // per thread
    __syncthreads();
    const int wper = (words + kBuildThreads - 1) / kBuildThreads;
    const int w0 = min(words, tid * wper), w1 = min(words, w0 + wper);
    int c = 0;
    for (int w = w0; w < w1; ++w) c += __popc(mark[w]);
    part[tid] = c;
    __syncthreads();
    for (int off = 1; off < kBuildThreads; off <<= 1) {
        const int v = tid >= off ? part[tid - off] : 0;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    int r = part[tid] - c;
    for (int w = w0; w < w1; ++w) {
        first[(size_t)blockIdx.x * words + w] = mark[w];
        before[(size_t)blockIdx.x * words + w] = (uint16_t)r;
        r += __popc(mark[w]);
    }
}

constexpr int kTileThreads = 1024;   // one block per SM (192 KB of values)

// buf[pos[i]] = src[i], i < n.  Four at a time where both are aligned.
__device__ __forceinline__ void tile_in(const float *src, const uint16_t *pos, int n, float *buf)
{
    int i0 = 0;
    if (((reinterpret_cast<uintptr_t>(src) & 15u) | (reinterpret_cast<uintptr_t>(pos) & 7u)) == 0) {
        i0 = n & ~3;
#pragma unroll 4
        for (int i = threadIdx.x * 4; i < i0; i += blockDim.x * 4) {
            const float4 v = __ldcs(reinterpret_cast<const float4 *>(src + i));
            const ushort4 l = __ldcs(reinterpret_cast<const ushort4 *>(pos + i));
            buf[l.x] = v.x; buf[l.y] = v.y; buf[l.z] = v.z; buf[l.w] = v.w;
        }
    }
#pragma unroll 4
    for (int i = i0 + threadIdx.x; i < n; i += blockDim.x)
        buf[__ldcs(pos + i)] = __ldcs(src + i);
}

__global__ void __launch_bounds__(kTileThreads)
    tile_out_kernel(const float *src, const uint16_t *pos1, const uint32_t *first,
                    const uint16_t *before, const int32_t *run, float *stage, int64_t nnz, int W,
                    int tiles)
{
    // the tile's values, then its run tables (read from global memory where
    // they are used, 2 x slower: two dependent loads per store)
    extern __shared__ float buf[];
    uint32_t *fw = reinterpret_cast<uint32_t *>(buf + W);
    int32_t *rn = reinterpret_cast<int32_t *>(fw + W / 32);
    uint16_t *bw = reinterpret_cast<uint16_t *>(rn + tiles);
    const int tid = threadIdx.x, words = W / 32;
    const int64_t base = (int64_t)blockIdx.x * W;
    const int n = (int)min((int64_t)W, nnz - base);
    for (int w = tid; w < words; w += blockDim.x) {
        fw[w] = __ldcs(first + (size_t)blockIdx.x * words + w);
        bw[w] = __ldcs(before + (size_t)blockIdx.x * words + w);
    }
    for (int b = tid; b < tiles; b += blockDim.x)
        rn[b] = __ldcs(run + (size_t)blockIdx.x * tiles + b);
    tile_in(src + base, pos1 + base, n, buf);
    __syncthreads();
    const uint32_t upto = 0xffffffffu >> (31 - (tid & 31));   // this lane and those before
#pragma unroll 4
    for (int i = tid; i < n; i += blockDim.x) {
        const int o = (int)bw[i / 32] + __popc(fw[i / 32] & upto) - 1;
        stage[i + rn[o]] = buf[i];
    }
}

__global__ void __launch_bounds__(kTileThreads)
    tile_sort_kernel(const float *stage, const uint16_t *pos2, float *dst, int64_t nnz, int W)
{
    extern __shared__ float buf[];
    const int64_t base = (int64_t)blockIdx.x * W;
    const int n = (int)min((int64_t)W, nnz - base);
    tile_in(stage + base, pos2 + base, n, buf);
    __syncthreads();
    const int n4 = n & ~3;   // dst + base is 16-byte aligned (W is a multiple of 4)
    for (int i = threadIdx.x * 4; i < n4; i += blockDim.x * 4)
        *reinterpret_cast<float4 *>(dst + base + i) = *reinterpret_cast<const float4 *>(buf + i);
    for (int i = n4 + threadIdx.x; i < n; i += blockDim.x)
        dst[base + i] = buf[i];
}

// Shared memory of pass 1: the values and the run tables.
size_t out_shared(int W, int tiles)
{
    return sizeof(float) * (size_t)W + (size_t)(W / 32) * 6 + sizeof(int32_t) * (size_t)tiles;
}
static_assert(sizeof(float) * kTileValuesMax + kTileValuesMax / 32 * 6 + 4 * kTilesMax <= 227 * 1024,
              "pass 1 at its largest");

// Raises both kernels' limit of dynamic shared memory, once per device (a bit
// per device of the first 64).
cudaError_t allow_shared()
{
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (bit && (done.load() & bit))
        return cudaSuccess;
    e = cudaFuncSetAttribute(tile_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)out_shared(kTileValuesMax, kTilesMax));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tile_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kTileValuesMax * (int)sizeof(float));
    if (e == cudaSuccess)
        done.fetch_or(bit);
    return e;
}

}  // namespace

// Below 2^24 values a single gather finds them in L2 (8.4M values: 43 us either
// way; 3.9M: 19 against 24); above 2^28 runs get short and their table large.
int32_t values_tile(int64_t nnz)
{
    return nnz > (int64_t(1) << 24) && nnz <= (int64_t(1) << 28) ? kTileValuesMax : 0;
}

cudaError_t build_value_tiles(ValueTiles &v, const int32_t *perm, int64_t nnz, uint32_t *inv,
                              cudaStream_t st)
{
    const int W = v.W, tiles = v.tiles;
    const unsigned grid = (unsigned)std::min<int64_t>((nnz + 255) / 256, (int64_t)sm_count() * 32);
    const size_t shared = sizeof(int32_t) * (size_t)tiles;
    inverse_kernel<<<grid, 256, 0, st>>>(perm, nnz, inv);
    run_count_kernel<<<tiles, 512, shared, st>>>(inv, nnz, W, tiles, v.run);
    run_place_kernel<<<(tiles + 127) / 128, 128, 0, st>>>(W, tiles, v.run);
    tile_places_kernel<<<tiles, kBuildThreads, shared, st>>>(inv, nnz, W, tiles, v.run, v.pos1, v.pos2,
                                                             v.first, v.before);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? allow_shared() : e;
}

cudaError_t launch_value_tiles(const ValueTiles &v, const float *src, float *dst, int64_t nnz,
                               cudaStream_t st)
{
    tile_out_kernel<<<v.tiles, kTileThreads, out_shared(v.W, v.tiles), st>>>(
        src, v.pos1, v.first, v.before, v.run, v.stage, nnz, v.W, v.tiles);
    tile_sort_kernel<<<v.tiles, kTileThreads, sizeof(float) * (size_t)v.W, st>>>(v.stage, v.pos2, dst,
                                                                               nnz, v.W);
    return cudaGetLastError();
}

}  // namespace fmm
