// fmm_fusedmm_noalloc: FusedMMA without a plan and without any allocation.
//
// Some callers cannot allocate device memory at the point where they need
// the product: code running inside a memory pool or arena that owns all of
// the device memory, a runtime that forbids cudaMalloc (and the implicit
// synchronisation it can cause) on its hot path, or a host library that is
// handed only its inputs and outputs.  fmm_plan_create allocates (S^T, the
// schedule, the partial rows), so those callers cannot use a plan.  This
// entry point computes the same FusedMMA as fmm_fusedmm from the CSR
// directly.  Its only scratch memory -- the chunk list and partial rows of
// long rows -- lives in the file-scope device array below, of fixed size.
//
// The passes are those a plan picks by default, compiled with the checks that
// a pattern no plan has validated needs.  What a plan prepares for
// them is prepared on every call: the work items of the rows in order of
// length, which one kernel counts per length key and another places (one block
// does both for few rows; the order within a key is free: a row's result does
// not depend on it).  With
// rows of any lengths side by side, a warp and its block wait for their
// longest row, which costs far more: Zipf(1.2) rows, 200003 x 100003, 4.8M
// nonzeros, r = 128, bfloat16 (GB300), 810 us with the rows in the caller's
// order in blocks of 16 rows, 412 with lane groups sharing a row and chunks of
// 128, 198 in order of length (counting and placing 17, the pass 173).
//
// Scratch:  g_noalloc_scratch, 34,603,264 bytes per device (every device that
// loads this library's module holds it until the process exits):
//   header    2304 B          counters: chunks, split rows, rows per length
//                             key and rows placed per length key
//   chunks    up to 64 Ki x 16 B  work item of each chunk of a long row
//   split     as many x 16 B  (row, first chunk, chunk count) of each long row
//   items     up to 1 Mi x 16 B  work items of a slab of rows
//   partials  the rest        one partial output row per chunk
// The header and the chunk slots in use are cleared at the start of a slab (of
// the header one block for few rows uses, and sets, the split rows alone).
// More than 2^20 rows go slab by slab.  Rows longer than ch nonzeros are split
// into chunks of ch, where ch = max(128, ceil(2 nnz / cap)) and cap = the
// partial rows there is room for, 64 Ki at most: every long row has more than
// ch nonzeros, so its ceil(deg / ch) chunks number fewer than 2 deg / ch, and
// all chunks together fewer than 2 nnz / ch <= cap.  The partial rows of a
// long row are summed in chunk order, so results are deterministic.  r may be
// at most 65536 (FMM_EOVERFLOW otherwise).
//
// Every call uses the same array: calls that overlap on the GPU (two streams,
// or two host threads without ordering) race on it and give wrong results.
// Order them on one stream.  Every call looks up the array's device address
// with cudaGetSymbolAddress on the current device (no allocation); the first
// call on a device may load the library's module there, so make that first
// call before any stream capture.
#include <algorithm>
#include <cstdio>

#include "fmm_flex.cuh"
#include "fmm_pipe.cuh"
#include "fmm_staged.cuh"

namespace fmm {
namespace noalloc {

constexpr int32_t MAX_CHUNKS = 1 << 16;
constexpr int32_t MAX_SLAB = 1 << 20;
constexpr int32_t MAX_R = 1 << 16;
constexpr int32_t MIN_CHUNK = 128;
constexpr size_t SCRATCH_BYTES = 34603264;

struct Header {
    int32_t n_chunks;
    int32_t n_split;
    int32_t pad[62];
    int32_t rows[256];      // rows per length key
    int32_t placed[256];    // of them, placed
};
constexpr size_t CHUNKS_OFF = sizeof(Header);
static_assert(CHUNKS_OFF % 256 == 0, "alignment");

static __device__ __align__(256) unsigned char g_noalloc_scratch[SCRATCH_BYTES];

struct Args {
    const int32_t *row_ptr;
    int32_t first, rows;    // the slab's rows
    int32_t ch;             // nonzeros per chunk
    int32_t cap;            // chunk slots (and split entries)
    int32_t r;
    int64_t nnz;
    Header *hdr;
    int4 *items;            // cap chunk slots, then the rows
    int4 *split;
};

// Row range of `row`, or an empty range if row_ptr is not consistent there
// (memory safety only: results for malformed patterns are unspecified).
__device__ __forceinline__ int2 row_range(const Args &a, int row)
{
    const int beg = __ldg(a.row_ptr + row), end = __ldg(a.row_ptr + row + 1);
    return beg < 0 || end < beg || (int64_t)end > a.nnz ? make_int2(0, 0) : make_int2(beg, end);
}

constexpr int kBlock = 256;
constexpr int kPerThread = 4;   // rows per thread of the two setup kernels

// Counts the slab's rows per length key (key 0: long rows) and lists the
// chunks of the long ones.
__global__ void __launch_bounds__(kBlock) count_kernel(const Args a)
{
    __shared__ int32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int t = 0; t < kPerThread; ++t) {
        const int64_t i = (int64_t)blockIdx.x * (kBlock * kPerThread) + t * kBlock + threadIdx.x;
        const int row = a.first + (int)i;
        int2 p = make_int2(0, 0);
        int nc = 0;   // chunks of this lane's row
        if (i < a.rows) {
            p = row_range(a, row);
            const uint32_t key = length_key(p.y - p.x, a.ch);
            atomicAdd(&cnt[key], 1);
            if (key == 0)
                nc = (int)(((int64_t)p.y - p.x + a.ch - 1) / a.ch);
        }
        // the warp takes its chunk slots and split entries at once
        const unsigned is_long = __ballot_sync(0xffffffffu, nc > 0);
        if (!is_long)
            continue;
        int upto = nc;   // chunks of lanes 0 ... lane
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, upto, off);
            if (lane >= off) upto += o;
        }
        int first = 0, slot = 0;
        if (lane == 31) {
            first = atomicAdd(&a.hdr->n_chunks, upto);
            slot = atomicAdd(&a.hdr->n_split, __popc(is_long));
        }
        first = __shfl_sync(0xffffffffu, first, 31) + upto - nc;
        slot = __shfl_sync(0xffffffffu, slot, 31) + __popc(is_long & ((1u << lane) - 1u));
        if (nc == 0 || slot >= a.cap)
            continue;   // (a full table: only a malformed pattern)
        const bool fits = first >= 0 && (int64_t)first + nc <= a.cap;
        a.split[slot] = make_int4(row, fits ? first : 0, fits ? nc : 0, 0);
        for (int c = 0; fits && c < nc; ++c) {
            const int64_t q = p.x + (int64_t)c * a.ch;
            a.items[first + c] = make_int4(row, (int)q, (int)min((int64_t)p.y, q + a.ch), 1);
        }
    }
    __syncthreads();
    if (cnt[threadIdx.x])
        atomicAdd(&a.hdr->rows[threadIdx.x], cnt[threadIdx.x]);
}

// Places the slab's rows in order of their length key.  A block ranks its
// rows per key in shared memory and takes its places of a key at once.
__global__ void __launch_bounds__(kBlock) place_kernel(const Args a)
{
    __shared__ int32_t cnt[256], base[256];
    const int tid = threadIdx.x;
    cnt[tid] = 0;
    const int mine = a.hdr->rows[tid];
    base[tid] = mine;
    __syncthreads();
    for (int off = 1; off < 256; off <<= 1) {   // inclusive scan of the key counts
        const int v = tid >= off ? base[tid - off] : 0;
        __syncthreads();
        base[tid] += v;
        __syncthreads();
    }
    const int start = base[tid] - mine;   // first place of key tid
    uint32_t key[kPerThread];
    int rank[kPerThread], row[kPerThread];
    int2 p[kPerThread];
#pragma unroll
    for (int t = 0; t < kPerThread; ++t) {
        const int64_t i = (int64_t)blockIdx.x * (kBlock * kPerThread) + t * kBlock + tid;
        row[t] = -1;
        if (i < a.rows) {
            row[t] = a.first + (int)i;
            p[t] = row_range(a, row[t]);
            key[t] = length_key(p[t].y - p[t].x, a.ch);
            rank[t] = atomicAdd(&cnt[key[t]], 1);
        }
    }
    __syncthreads();
    base[tid] = start + (cnt[tid] ? atomicAdd(&a.hdr->placed[tid], cnt[tid]) : 0);
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kPerThread; ++t)
        if (row[t] >= 0)   // a long row keeps its place, without work
            a.items[a.cap + base[key[t]] + rank[t]] =
                key[t] == 0 ? make_int4(0, 0, 0, 0) : make_int4(row[t], p[t].x, p[t].y, 1);
}

// Both steps in one block, for slabs of at most kSmallRows rows and kSmallSlots
// chunk slots: the counts stay in shared memory, so nothing is cleared before
// or read back between.  Lanes with one key take their places together (rows of
// one length would queue at a single counter).  Erdos-Renyi rows of 16, float32,
// r = 128, a call with the two kernels and the memset and this way: 300 rows 15.7
// and 9.5 us, 2000 rows 17.1 and 12.8; 4000 rows of 30 24.0 and 22.2.
constexpr int kSmallBlock = 1024;
constexpr int kSmallRows = kSmallBlock * kPerThread;
constexpr int kSmallSlots = 4096;

__global__ void __launch_bounds__(kSmallBlock) order_small_kernel(const Args a)
{
    __shared__ int32_t cnt[256], base[256], n_chunks, n_split;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 256) cnt[tid] = 0;
    if (tid == 0) n_chunks = n_split = 0;
    for (int i = tid; i < a.cap; i += kSmallBlock) a.items[i] = make_int4(0, 0, 0, 0);
    __syncthreads();
    uint32_t key[kPerThread];
    int rank[kPerThread], row[kPerThread];
    int2 p[kPerThread];
#pragma unroll
    for (int t = 0; t < kPerThread; ++t) {
        const int i = t * kSmallBlock + tid;
        row[t] = -1;
        p[t] = make_int2(0, 0);
        key[t] = 256;   // no row
        if (i < a.rows) {
            row[t] = a.first + i;
            p[t] = row_range(a, row[t]);
            key[t] = length_key(p[t].y - p[t].x, a.ch);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key[t]);
        const int leader = __ffs(peers) - 1;
        int at = 0;
        if (lane == leader && key[t] < 256)
            at = atomicAdd(&cnt[key[t]], __popc(peers));
        rank[t] = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
        if (key[t] != 0)
            continue;
        // a long row: its split entry and chunk slots (a full table: only a
        // malformed pattern)
        const int nc = (int)(((int64_t)p[t].y - p[t].x + a.ch - 1) / a.ch);
        const int first = atomicAdd(&n_chunks, nc), slot = atomicAdd(&n_split, 1);
        if (slot >= a.cap)
            continue;
        const bool fits = first >= 0 && (int64_t)first + nc <= a.cap;
        a.split[slot] = make_int4(row[t], fits ? first : 0, fits ? nc : 0, 0);
        for (int c = 0; fits && c < nc; ++c) {
            const int64_t q = p[t].x + (int64_t)c * a.ch;
            a.items[first + c] = make_int4(row[t], (int)q, (int)min((int64_t)p[t].y, q + a.ch), 1);
        }
    }
    __syncthreads();
    const int mine = tid < 256 ? cnt[tid] : 0;
    if (tid < 256) base[tid] = mine;
    __syncthreads();
    for (int off = 1; off < 256; off <<= 1) {   // inclusive scan of the key counts
        const int v = tid < 256 && tid >= off ? base[tid - off] : 0;
        __syncthreads();
        if (tid < 256) base[tid] += v;
        __syncthreads();
    }
    if (tid < 256) base[tid] -= mine;   // first place of key tid
    if (tid == 0) a.hdr->n_split = n_split;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kPerThread; ++t)
        if (row[t] >= 0)   // a long row keeps its place, without work
            a.items[a.cap + base[key[t]] + rank[t]] =
                key[t] == 0 ? make_int4(0, 0, 0, 0) : make_int4(row[t], p[t].x, p[t].y, 1);
}

// The pass over the work items: for vectorised widths the layouts of
// default_variant (the register ring for bfloat16 rows, the staged pass for
// float32 rows of r = 128, else the team kernel with 8 elements per lane),
// otherwise the flexible or the generic pass.
template <typename T, int R>
cudaError_t launch_width(const PassArgs &p, cudaStream_t st)
{
    constexpr int B = base_vpl<T, R>();
    constexpr int V = sizeof(T) == 4 && R * 4 / 16 <= 32 ? 2 * B : B;   // 8 elements per lane
    if constexpr (sizeof(T) == 2) {
        if ((reinterpret_cast<uintptr_t>(p.Y) & 31u) == 0)
            return launch_pipe<M_FUSED, T, R, 2 * B, 1, R == 128 ? 4 : 2, 2, 1, true>(p, st);
    }
    if constexpr (sizeof(T) == 4 && R == 128)
        return launch_staged<M_FUSED, T, R, V, 4, true>(p, st);
    else
        return launch_team<M_FUSED, T, R, V, 1, 2, true>(p, st);
}

template <typename T>
cudaError_t launch_checked(const PassArgs &p, int dtype, cudaStream_t st)
{
    const int vb = flex_vector_bytes(p, dtype);
    if (vb == 16) {
        switch (p.r) {
        case 32: return launch_width<T, 32>(p, st);
        case 64: return launch_width<T, 64>(p, st);
        case 128: return launch_width<T, 128>(p, st);
        case 256: return launch_width<T, 256>(p, st);
        default: break;
        }
    }
    if (p.r <= kFlexMaxR)
        return dispatch_flex<M_FUSED, T, false, true>(p, vb, flex_groups(p), st);
    const long long total = (long long)p.n_chunks + p.n_light;
    row_pass_generic<M_FUSED, T, true><<<(unsigned)((total + 7) / 8), 256, 0, st>>>(p);
    return cudaGetLastError();
}

// The array's device address, looked up on every call with the current
// device (cudaGetSymbolAddress allocates nothing).  Nothing is cached, so a
// module reloaded at another address (after cudaDeviceReset) is followed.
int scratch_base(unsigned char **base)
{
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
        set_error("cudaGetSymbolAddress(no-alloc scratch)", e);
        return FMM_ECUDA;
    }
    *base = static_cast<unsigned char *>(p);
    return FMM_OK;
}

}  // namespace noalloc
}  // namespace fmm

extern "C" int fmm_fusedmm_noalloc(const fmm_csr *S, int32_t r, int32_t dtype, const float *vals,
                                   const void *A, const void *B, float *out_m, fmm_stream stream)
{
    using namespace fmm;
    using namespace fmm::noalloc;
    int rc = check_csr_args(S);
    if (rc)
        return rc;
    if (r < 1 || (dtype != FMM_F32 && dtype != FMM_BF16)) {
        set_error_msg("r must be >= 1 and dtype FMM_F32 or FMM_BF16");
        return FMM_EUNSUPPORTED;
    }
    if (r > MAX_R) {
        set_error_msg("r exceeds the no-alloc maximum of 65536");
        return FMM_EOVERFLOW;
    }
    if ((S->m > 0 && (!A || !out_m)) || (S->n > 0 && !B)) {
        set_error_msg("A, B or out_m is NULL");
        return FMM_EINVAL;
    }
    if (S->m == 0)
        return FMM_OK;
    unsigned char *base = nullptr;
    rc = scratch_base(&base);
    if (rc)
        return rc;
    // chunk slots: as many as there is room for beside the items of a slab
    // (a split entry, an item and a partial row each), at most MAX_CHUNKS
    const int64_t slab = std::min<int64_t>(S->m, MAX_SLAB);
    const int64_t room = (int64_t)(SCRATCH_BYTES - CHUNKS_OFF) - 16 * slab - 256;
    const int64_t cap = std::min<int64_t>(MAX_CHUNKS, room / (2 * (int64_t)sizeof(int4) + 4 * (int64_t)r));
    const int64_t ch = std::max<int64_t>(MIN_CHUNK, (2 * S->nnz + cap - 1) / cap);
    Args a;
    a.row_ptr = S->row_ptr;
    a.ch = (int32_t)std::min<int64_t>(ch, INT32_MAX);
    // slots that this pattern can use
    a.cap = (int32_t)std::min<int64_t>(cap, 2 * S->nnz / a.ch);
    a.r = r;
    a.nnz = S->nnz;
    a.hdr = reinterpret_cast<Header *>(base);
    a.items = reinterpret_cast<int4 *>(base + CHUNKS_OFF);
    a.split = a.items + a.cap + slab;
    float *partials = reinterpret_cast<float *>(a.split + a.cap);
    partials += (-(reinterpret_cast<uintptr_t>(partials) / 4)) & 63;   // 256-byte aligned
    PassArgs p{};
    p.row_ptr = S->row_ptr;
    p.col_idx = S->col_idx;
    p.items = a.items;
    p.n_chunks = a.cap;
    p.partials = partials;
    p.s = vals;
    p.s_direct = 1;
    p.L = A;
    p.Y = B;
    p.out = out_m;
    p.r = r;
    p.nnz = S->nnz;
    p.cols = S->n;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = cudaSuccess;
    for (int64_t first = 0; first < S->m && e == cudaSuccess; first += slab) {
        a.first = (int32_t)first;
        a.rows = (int32_t)std::min<int64_t>(slab, S->m - first);
        p.n_light = a.rows;
        const unsigned blocks = (unsigned)((a.rows + kBlock * kPerThread - 1) / (kBlock * kPerThread));
        if (a.rows <= kSmallRows && a.cap <= kSmallSlots) {
            order_small_kernel<<<1, kSmallBlock, 0, st>>>(a);
        } else {
            e = cudaMemsetAsync(base, 0, CHUNKS_OFF + sizeof(int4) * (size_t)a.cap, st);
            if (e != cudaSuccess)
                break;
            count_kernel<<<blocks, kBlock, 0, st>>>(a);
            place_kernel<<<blocks, kBlock, 0, st>>>(a);
        }
        e = dtype == FMM_BF16 ? launch_checked<bf16_t>(p, dtype, st)
                              : launch_checked<float>(p, dtype, st);
        if (e == cudaSuccess && a.cap > 0) {
            // a long row has two chunks at least
            e = launch_combine(a.split, a.cap / 2 + 1, &a.hdr->n_split, partials, out_m, nullptr, r,
                               false, st);
        }
        if (e == cudaSuccess)
            e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error("fmm_fusedmm_noalloc launch", e);
        return FMM_ECUDA;
    }
    return FMM_OK;
}
