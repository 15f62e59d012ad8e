// Batched FusedMM: many uneven matrices in one persistent launch.
//
// Every matrix of a batch keeps its own plan (pattern, S^T, row order).  A
// batch lists, for each matrix and each row pass of a phase, work units of
// consecutive teams (chunks, then rows in the plan's longest-first order).  The
// units are handed out by a device counter: every warp of a grid sized to fill
// the GPU pops a unit, runs the pass body of that matrix's row width and layout
// on it, and pops the next, until the list is empty.  There is a list, a counter
// and a persistent kernel for the team layouts of each phase and for the
// register-ring layouts of each role, so forward (FusedMMA of every matrix) is
// one launch or two, backward (dA and ds over S, dB over S^T) up to three; a
// last kernel sums partial rows.  The counters are cleared by a memset queued
// before each phase, so both can be captured in a CUDA graph and replayed.
//
// Plans whose split_nnz set no limit take rows above the default split size in
// chunks, here as in their own calls, with partial rows in the batch's own
// memory, summed in chunk order.  Results are bitwise those of the per-matrix
// calls: the layouts are those of the plan, and the passes that a call may take
// in their place (fmm_wide.cuh) keep their order of sums.
//
// Units are handed out matrix by matrix, the matrices with the most work
// first, and inside a matrix chunks first and then the longest rows: the
// rows gathered by the warps running at one time are then those of one or a
// few matrices, which fit L2 (a matrix of 2 10^5 rows at r = 128 in bfloat16
// gathers from 51 MB), while the order over all matrices at once gathers
// from gigabytes.  The last matrices are the smallest, so the launch still
// ends evenly.  64 matrices, rows log-uniform in [1e3, 2e5], r of 32, 64 and
// 128, bfloat16 (GB300): forward 4.08 -> 1.97 ms, backward 7.71 -> 6.09, with
// the rows above the default size cut into chunks; uncut, the hub row of the
// largest matrix alone took the 4.08 ms.  With the register-ring layouts, the
// pass arguments in shared memory and smaller units 1.36 and 5.21 ms.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "fmm_pipe.cuh"

namespace fmm {

struct BatchItemDev {
    PassArgs fwd;       // over S: FusedMMA
    PassArgs bwd_row;   // over S: dA (and ds)
    PassArgs bwd_col;   // over S^T: dB
};

// 128 columns (or fewer) of one split row: the sum of `chunks` partial rows,
// r floats apart, in chunk order.
struct BatchSum {
    const float *partials;
    float *out;
    int32_t chunks, cols, r;
};

__global__ void __launch_bounds__(128) batch_sum_kernel(const BatchSum *sums, int n)
{
    constexpr int LOADS = 16;   // partial rows loaded before their additions
    const int w = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (w >= n)
        return;
    const BatchSum s = sums[w];
    const int k = (threadIdx.x & 31) * 4;
    if (k >= s.cols)
        return;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < s.chunks; c0 += LOADS) {
        float4 x[LOADS];
#pragma unroll
        for (int i = 0; i < LOADS; ++i)
            if (c0 + i < s.chunks)
                x[i] = __ldcs(reinterpret_cast<const float4 *>(s.partials + (size_t)(c0 + i) * s.r + k));
#pragma unroll
        for (int i = 0; i < LOADS; ++i)
            if (c0 + i < s.chunks) {
                acc.x += x[i].x; acc.y += x[i].y; acc.z += x[i].z; acc.w += x[i].w;
            }
    }
    *reinterpret_cast<float4 *>(s.out + k) = acc;
}

enum UnitKind { U_FWD = 0, U_BWD_ROW = 1, U_BWD_COL = 2 };

// Work items [begin, begin + count) of pass `a` (chunks of its split rows,
// then rows in plan order).
template <int MODE, typename T, int R, int VPL, int NG, int U>
__device__ __forceinline__ void run_unit(const PassArgs &a, int begin, int count)
{
    constexpr int TEAM = TeamShape<T, R, VPL, NG>::TEAM;
    constexpr int TPW = 32 / TEAM;
    const int lane = threadIdx.x & 31;
    for (int t0 = 0; t0 < count; t0 += TPW) {
        const int t = t0 + lane / TEAM;
        team_pass_body<MODE, T, R, VPL, NG, U, false, false>(a, (long long)begin + t, t < count);
    }
}

// The variant codes a batch can run: one kernel holds every (width, code)
// path, and its register count is the largest path's, so batches take only
// light variants: at most 32 floats live per lane in the forward phase (64
// registers, 4 blocks per SM; with 48 it needed 80 and ran 19 % slower on
// the 512-matrix batch) and 48 in the backward phase, whose pass over S^T
// holds two gathered rows per nonzero.
template <int MODE, typename T>
constexpr bool batch_code_ok(int r, int code)
{
    const int vecs = r * (int)sizeof(T) / 16;
    const int base = vecs > 32 ? vecs / 32 : 1;
    const int V = (code / 100) * base, N = (code / 10) % 10, UU = code % 10;
    if (V < 1 || vecs % V != 0) return false;
    const int g = vecs / V;
    const int E = V * (16 / (int)sizeof(T));
    const int live = E * (UU * (MODE == M_BWD_COL ? 2 : 1) + 2 + (MODE == M_BWD_ROW ? 1 : 0));
    return g >= 1 && (g & (g - 1)) == 0 && g * N <= 32 && 32 % (g * N) == 0 &&
           live <= (MODE == M_FUSED ? 32 : 48);
}

template <int MODE, typename T>
__device__ __forceinline__ void run_code(int code, const PassArgs &a, int begin, int count)
{
#define FMM_BATCH_CASE(RR, M, N, UU)                                                         \
    case (RR << 16) | (M * 100 + N * 10 + UU):                                               \
        if constexpr (batch_code_ok<MODE, T>(RR, M * 100 + N * 10 + UU))                    \
            run_unit<MODE, T, RR, M * base_vpl<T, RR>(), N, UU>(a, begin, count);            \
        return;
#define FMM_BATCH_R(RR)                                                                      \
    FMM_BATCH_CASE(RR, 1, 1, 2) FMM_BATCH_CASE(RR, 1, 1, 4) FMM_BATCH_CASE(RR, 1, 2, 2)     \
    FMM_BATCH_CASE(RR, 2, 1, 2) FMM_BATCH_CASE(RR, 2, 1, 4) FMM_BATCH_CASE(RR, 2, 2, 1)
    switch (code) {
        FMM_BATCH_R(32)
        FMM_BATCH_R(64)
        FMM_BATCH_R(128)
        FMM_BATCH_R(256)
    default: return;
    }
#undef FMM_BATCH_R
#undef FMM_BATCH_CASE
}

// Items of plans left to their own choice: the ring layouts of role_variant, in
// a kernel of their own (128 registers a thread, which the team codes above
// would only pay for).
template <int MODE, typename T, int R, int VPL, int RING>
__device__ __forceinline__ void run_ring_unit(const PassArgs &a, int begin, int count)
{
    constexpr int G = TeamShape<T, R, VPL, 1>::G, TPW = 32 / G;
    const int lane = threadIdx.x & 31;
    for (int t0 = 0; t0 < count; t0 += TPW) {
        const int t = t0 + lane / G;
        pipe_pass_body<MODE, T, R, VPL, 1, RING, 1, false>(a, (long long)begin + t, t < count);
    }
}

constexpr int kRingCode = 9;   // in place of a team code

// Whether the own choice of a pass over `side` is a layout of the ring kernels
// below (the adjoint over S^T of bfloat16 r = 32 by the team body).
bool ring_role(int mode, int dtype, int r, const Side &side, int64_t nnz)
{
    if (dtype == FMM_F32 && (mode != M_BWD_ROW || r != 256))
        return false;
    if (mode == M_BWD_COL && r == 32)
        return true;
    const long long items = std::max<long long>(1, (long long)side.n_chunks + side.n_light);
    return role_variant(mode, r, dtype, (double)nnz / items, side.longest).ring > 0;
}

// Vectors per lane of the ring layouts of bfloat16 rows (0: the team kernel).
template <int MODE>
constexpr int ring_vpl(int r)
{
    return MODE != M_BWD_COL ? 2 : r == 32 ? 0 : r == 64 ? 1 : 2;
}
template <int MODE>
constexpr int ring_depth(int r)
{
    return MODE == M_FUSED ? (r == 128 ? 4 : 2) : MODE == M_BWD_ROW ? 4 : r == 64 ? 4 : 2;
}

template <int MODE, typename T>
__device__ __forceinline__ void run_ring(int r, const PassArgs &a, int begin, int count)
{
    if constexpr (sizeof(T) == 4) {   // (r = 256)
        run_ring_unit<MODE, T, 256, 2 * base_vpl<T, 256>(), 2>(a, begin, count);
    } else {
#define FMM_RING_R(RR)                                                                       \
    case RR:                                                                                 \
        run_ring_unit<MODE, T, RR, ring_vpl<MODE>(RR), ring_depth<MODE>(RR)>(a, begin, count); \
        return;
        switch (r) {
        case 32:
            if constexpr (ring_vpl<MODE>(32) == 0)
                run_unit<MODE, T, 32, 1, 1, 2>(a, begin, count);
            else
                run_ring_unit<MODE, T, 32, ring_vpl<MODE>(32), ring_depth<MODE>(32)>(a, begin, count);
            return;
        FMM_RING_R(64) FMM_RING_R(128) FMM_RING_R(256)
        }
#undef FMM_RING_R
    }
}

// Hands the units of a list to the calling warp until none are left.  The next
// unit's number is fetched while the current unit is worked on, and the pass
// of the current matrix is kept in shared memory (one PassArgs per warp),
// where it costs no registers: read from global memory by the row, it cost the
// forward phase of the 64-matrix batch 1.72 ms in place of 1.41.
template <typename Work>
__device__ __forceinline__ void for_units(const BatchItemDev *items, const int4 *units, int n_units,
                                          int *counter, unsigned char *shared, Work work)
{
    static_assert(sizeof(PassArgs) % 8 == 0, "copied in 8-byte words");
    constexpr int WORDS = sizeof(PassArgs) / 8;
    const PassArgs &pass = *reinterpret_cast<const PassArgs *>(shared);
    const int lane = threadIdx.x & 31;
    int next = 0, item = -1;
    if (lane == 0)
        next = atomicAdd(counter, 1);
    for (;;) {
        const int u = __shfl_sync(0xffffffffu, next, 0);
        if (u >= n_units)
            break;
        if (lane == 0)
            next = atomicAdd(counter, 1);
        const int4 unit = __ldg(units + u);
        const int kind = unit.y & 3, code = unit.y >> 2;
        if (unit.x * 4 + kind != item) {   // uniform in the warp
            item = unit.x * 4 + kind;
            const BatchItemDev &it = items[unit.x];
            const PassArgs &role = kind == U_FWD ? it.fwd : kind == U_BWD_ROW ? it.bwd_row : it.bwd_col;
            const uint2 *from = reinterpret_cast<const uint2 *>(&role);
            __syncwarp();
            for (int w = lane; w < WORDS; w += 32) reinterpret_cast<uint2 *>(shared)[w] = from[w];
            __syncwarp();
        }
        work(kind, code, pass, unit.z, unit.w);
    }
}

// The ring layouts have a kernel per role: one for the whole backward phase
// spilled at its 128 registers (6.2 ms in place of 1.86 + 3.6).
template <int MODE, typename T>
__global__ void __launch_bounds__(32, 16) ring_batch_kernel(const BatchItemDev *items,
                                                            const int4 *units, int n_units,
                                                            int *counter)
{
    __shared__ __align__(16) unsigned char shared[sizeof(PassArgs)];
    for_units(items, units, n_units, counter, shared,
              [](int, int, const PassArgs &a, int begin, int count) {
                  run_ring<MODE, T>(a.r, a, begin, count);
              });
}

// The team layouts one per phase: a kernel per role was slower (48 float32
// matrices of 1e3 to 9e3 rows, a step 1.08 -> 1.36 ms; the rows of one matrix
// are then gathered by both passes close together, and one launch fewer ends
// unevenly).
template <typename T, int PHASE>
__global__ void __launch_bounds__(256) batch_kernel(const BatchItemDev *items, const int4 *units,
                                                    int n_units, int *counter)
{
    __shared__ __align__(16) unsigned char shared[8][(sizeof(PassArgs) + 15) / 16 * 16];
    for_units(items, units, n_units, counter, shared[threadIdx.x >> 5],
              [](int kind, int code, const PassArgs &a, int begin, int count) {
                  if constexpr (PHASE == 0) {
                      run_code<M_FUSED, T>(code, a, begin, count);
                  } else {
                      if (kind == U_BWD_ROW)
                          run_code<M_BWD_ROW, T>(code, a, begin, count);
                      else
                          run_code<M_BWD_COL, T>(code, a, begin, count);
                  }
              });
}

template <typename T>
bool batch_supported(int mode, int r, int code)
{
    switch (mode) {
    case M_FUSED: return batch_code_ok<M_FUSED, T>(r, code);
    case M_BWD_ROW: return batch_code_ok<M_BWD_ROW, T>(r, code);
    default: return batch_code_ok<M_BWD_COL, T>(r, code);
    }
}

// Codes a batch accepts (the FMM_BATCH_R list below).
inline bool batch_listed(int code)
{
    return code == 112 || code == 114 || code == 122 || code == 212 || code == 214 || code == 221;
}

}  // namespace fmm

using namespace fmm;

constexpr int LISTS = 5;   // of work units: a kernel and a counter each

struct fmm_batch {
    int32_t count = 0, dtype = 0, device = 0;
    bool has_bwd = false;
    BatchItemDev *d_items = nullptr;
    // units {item, 4 ((r << 16) | code) + kind, first work item, count} by list:
    // the team kernels' by phase, then the ring kernels' by kind
    int4 *d_units[LISTS] = {};
    int32_t n_units[LISTS] = {};
    int *d_counters = nullptr;
    float *d_partials = nullptr;            // partial rows of chunks, every pass its own
    BatchSum *d_sums_fwd = nullptr, *d_sums_bwd = nullptr;
    int32_t n_sums_fwd = 0, n_sums_bwd = 0;
    int grid[LISTS] = {};
};

namespace {

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool aligned32(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }

// The variant a batch runs for a pass: the plan's, if the batch kernels
// have it for this width and role, else the width's default.
int batch_code(int dtype, int mode, int r, const KernelVariant &v)
{
    const int want = encode_variant(v);
    const bool ok = batch_listed(want) &&
                    (dtype == FMM_BF16 ? batch_supported<bf16_t>(mode, r, want)
                                       : batch_supported<float>(mode, r, want));
    if (ok)
        return want;
    // the default team layout of the width (the batch kernels run the team
    // pass only), with fewer nonzeros per batch if needed
    KernelVariant d = team_default_variant(r, dtype);
    for (int u : {d.u, 2, 1}) {
        d.u = u;
        const int c = encode_variant(d);
        const bool dok = dtype == FMM_BF16 ? batch_supported<bf16_t>(mode, r, c)
                                           : batch_supported<float>(mode, r, c);
        if (dok)
            return c;
    }
    return 112;
}

// Teams per warp of a variant code at width r.
int teams_per_warp(int dtype, int r, int code, int mode)
{
    if (code == kRingCode && dtype == FMM_F32)
        return 2;   // 16 lanes, r = 256
    if (code == kRingCode) {
        const int vpl = mode == M_BWD_COL ? ring_vpl<M_BWD_COL>(r) : ring_vpl<M_FUSED>(r);
        return 32 / (r / 8 / std::max(1, vpl));
    }
    const int vecs = r * (dtype == FMM_BF16 ? 2 : 4) / 16;
    const int base = vecs > 32 ? vecs / 32 : 1;
    const int V = (code / 100) * base, N = (code / 10) % 10;
    return 32 / ((vecs / V) * N);
}

// Units of one pass: consecutive chunks, or consecutive rows within one
// length bucket, about unit_nnz nonzeros of work each (from the bucket's
// shortest row length), a multiple of the warp's team count.  Small units end
// a launch evenly (48 float32 matrices of 1e3 to 9e3 rows, forward + backward:
// units of 512 nonzeros 1120 us, 128: 770, 32: 631; the 64-matrix batch 6.89
// ms, 6.57, 6.59), but a list of them is a table of 16 bytes each, so
// fmm_batch_create aims at 2^19 units per role.
void make_units(std::vector<int4> &out, const Side &side, int item, int code, int tpw, int unit_nnz)
{
    for (int c = 0; c < side.n_chunks; c += tpw)
        out.push_back(make_int4(item, code, c, std::min(tpw, side.n_chunks - c)));
    for (int key = 1; key < 256; ++key) {   // key 0: the split rows
        const int b0 = side.bucket_start[key], b1 = side.bucket_start[key + 1];
        if (b1 <= b0)
            continue;
        int per = tpw;
        if (key >= 136 && key < 255) {
            const int lo = length_key_min((uint32_t)key);
            per = std::max(tpw, std::min(256, unit_nnz / std::max(lo, 1)));
            per = (per + tpw - 1) / tpw * tpw;
        } else if (key == 255) {
            per = 256;                        // empty rows: zero fills
        }
        const int shift = side.n_chunks - side.n_split;   // row position -> work item
        for (int t = b0; t < b1; t += per)
            out.push_back(make_int4(item, code, shift + t, std::min(per, b1 - t)));
    }
}

// The rows in chunks of one pass as (partial rows, output row, chunks) for
// batch_sum_kernel; passes without an output have none.
void make_sums(std::vector<BatchSum> &out, const Side &side, const float *partials, float *dst,
               int32_t r)
{
    if (!dst)
        return;
    for (const int4 &sp : side.split_host)
        for (int32_t k = 0; k < r; k += 128)
            out.push_back({partials + (size_t)sp.y * r + k, dst + (size_t)sp.x * r + k, sp.z,
                           std::min(128, r - k), r});
}

int grid_for(const void *kernel, int threads)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0);
    return std::max(1, sms * std::max(1, per));
}

#define CHECK(x)              \
    do {                      \
        int _rc = (x);        \
        if (_rc) return _rc;  \
    } while (0)

}  // namespace

extern "C" {

int fmm_plan_set_variant(fmm_plan *p, int32_t variant, int32_t variant_t)
{
    if (!p || (variant && !variant_known(variant)) || (variant_t && !variant_known(variant_t))) {
        set_error_msg("invalid plan or variant code");
        return FMM_EINVAL;
    }
    // the code of the plan's own choice gives a side that choice back (as a
    // layout of its own the code can be given to fmm_plan_create): a tuner that
    // times a code on both sides and keeps it on one keeps what it timed
    const KernelVariant own = default_variant(p->r, p->dtype, 0.0);
    auto of = [&](int32_t code) { return code == encode_variant(own) ? own : decode_variant(code); };
    if (variant)
        p->rows.variant = of(variant);
    if (variant_t)
        p->cols.variant = of(variant_t);
    return FMM_OK;
}

int fmm_batch_create(const fmm_batch_item *items, int32_t count, fmm_stream stream,
                     fmm_batch **batch)
{
    if (!batch || !items || count < 1) {
        set_error_msg("fmm_batch_create: NULL argument or empty batch");
        return FMM_EINVAL;
    }
    *batch = nullptr;
    const int dtype = items[0].plan ? items[0].plan->dtype : -1;
    int dev = -1;
    cudaGetDevice(&dev);
    bool bwd = true;
    for (int i = 0; i < count; ++i) {
        const fmm_batch_item &it = items[i];
        const fmm_plan *p = it.plan;
        if (!p || p->dtype != dtype || p->device != dev) {
            set_error_msg("batch items need plans of one dtype on the current device");
            return FMM_EINVAL;
        }
        if (!fast_r(p->r)) {
            set_error_msg("batch items need r in {32, 64, 128, 256}");
            return FMM_EUNSUPPORTED;
        }
        if (!p->no_limit && (p->rows.n_split || (p->has_t && p->cols.n_split))) {
            set_error_msg("batch plans must have no split rows (create them with a large split_nnz)");
            return FMM_EUNSUPPORTED;
        }
        const void *ptrs[] = {it.A, it.B, it.out, it.G, it.dA, it.dB};
        for (const void *q : ptrs)
            if (!aligned16(q)) {
                set_error_msg("batch dense operands must be 16-byte aligned");
                return FMM_EUNSUPPORTED;
            }
        if ((p->m > 0 && (!it.A || !it.out)) || (p->n > 0 && !it.B)) {
            set_error_msg("batch item without A, B or out");
            return FMM_EINVAL;
        }
        if (!it.G || (!it.dA && !it.dB && !it.ds) || (it.dB && !p->has_t))
            bwd = false;
    }
    fmm_batch *b = new fmm_batch();
    b->count = count;
    b->dtype = dtype;
    b->device = dev;
    b->has_bwd = bwd;
    cudaError_t e = cudaSuccess;
    // partial rows: forward, adjoint over S and adjoint over S^T of each item
    size_t partial_floats = 0;
    for (int i = 0; i < count; ++i) {
        const fmm_plan *p = items[i].plan;
        partial_floats += (size_t)p->r * ((bwd ? 2 : 1) * (size_t)p->rows.n_chunks +
                                          (bwd && items[i].dB ? (size_t)p->cols.n_chunks : 0));
    }
    if (partial_floats)
        e = cudaMalloc(&b->d_partials, sizeof(float) * partial_floats);
    if (e != cudaSuccess) {
        set_error("fmm_batch_create", e);
        fmm_batch_destroy(b);
        return e == cudaErrorMemoryAllocation ? FMM_ENOMEM : FMM_ECUDA;
    }
    float *next_partials = b->d_partials;
    int64_t total_nnz = 0;
    for (int i = 0; i < count; ++i) total_nnz += items[i].plan->nnz;
    const int unit_nnz = (int)std::min<int64_t>(512, std::max<int64_t>(32, total_nnz >> 19));
    // matrices in the order of their work, most first
    std::vector<int> order(count);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        return items[x].plan->nnz * items[x].plan->r > items[y].plan->nnz * items[y].plan->r;
    });
    std::vector<BatchItemDev> host(count);
    std::vector<int4> units[LISTS];
    std::vector<BatchSum> sums_f, sums_b;
    for (int i : order) {
        const fmm_batch_item &it = items[i];
        const fmm_plan *p = it.plan;
        BatchItemDev &d = host[i];
        auto fill = [&](PassArgs &a, const Side &side, const float *s, const void *L,
                        const void *Y, const float *H, float *out, float *nzout) {
            a.row_ptr = side.row_ptr;
            a.col_idx = side.col_idx;
            a.perm = side.perm;
            a.n_light = side.n_light;
            a.items = side.items;
            a.n_chunks = side.n_chunks;
            a.partials = next_partials;
            a.s = s;
            a.s_direct = 0;
            a.L = L;
            a.Y = Y;
            a.H = H;
            a.out = out;
            a.nzout = nzout;
            a.r = p->r;
        };
        fill(d.fwd, p->rows, it.vals, it.A, it.B, nullptr, it.out, nullptr);
        make_sums(sums_f, p->rows, next_partials, it.out, p->r);
        next_partials += (size_t)p->rows.n_chunks * p->r;
        fill(d.bwd_row, p->rows, it.vals, it.A, it.B, it.G, it.dA, it.ds);
        PassArgs empty{};
        d.bwd_col = empty;
        // the ring kernel loads gathered rows 32 bytes at a time
        auto code_of = [&](int mode, const Side &side, const void *Y, const void *H) {
            return side.variant.own && ring_role(mode, dtype, p->r, side, p->nnz) && aligned32(Y) &&
                           aligned32(H)
                       ? kRingCode
                       : batch_code(dtype, mode, p->r, side.variant);
        };
        auto list = [&](int kind, int code) -> std::vector<int4> & {
            return units[code == kRingCode ? 2 + kind : kind != U_FWD];
        };
        const int cf = code_of(M_FUSED, p->rows, it.B, nullptr);
        const int rcode = p->r << 16;
        make_units(list(U_FWD, cf), p->rows, i, 4 * (rcode | cf) + U_FWD, teams_per_warp(dtype, p->r, cf, M_FUSED),
                   unit_nnz);
        if (bwd) {
            const int cr = code_of(M_BWD_ROW, p->rows, it.B, nullptr);
            make_sums(sums_b, p->rows, next_partials, it.dA, p->r);
            next_partials += (size_t)p->rows.n_chunks * p->r;
            if (it.dA || it.ds)
                make_units(list(U_BWD_ROW, cr), p->rows, i, 4 * (rcode | cr) + U_BWD_ROW,
                           teams_per_warp(dtype, p->r, cr, M_BWD_ROW), unit_nnz);
            if (it.dB) {
                fill(d.bwd_col, p->cols, it.vals, it.B, it.A, it.G, it.dB, nullptr);
                make_sums(sums_b, p->cols, next_partials, it.dB, p->r);
                next_partials += (size_t)p->cols.n_chunks * p->r;
                const int cc = code_of(M_BWD_COL, p->cols, it.A, it.G);
                make_units(list(U_BWD_COL, cc), p->cols, i, 4 * (rcode | cc) + U_BWD_COL,
                           teams_per_warp(dtype, p->r, cc, M_BWD_COL), unit_nnz);
            }
        }
    }
    for (int k = 0; k < LISTS; ++k) b->n_units[k] = (int32_t)units[k].size();
    b->n_sums_fwd = (int32_t)sums_f.size();
    b->n_sums_bwd = (int32_t)sums_b.size();
    cudaStream_t st = (cudaStream_t)stream;
    // a device copy of a host table (at least one entry's room)
    auto upload = [&](auto **dst, const auto &v) {
        const size_t one = sizeof(v[0]);
        if (e == cudaSuccess)
            e = cudaMalloc((void **)dst, one * std::max<size_t>(1, v.size()));
        if (e == cudaSuccess && !v.empty())
            e = cudaMemcpyAsync(*dst, v.data(), one * v.size(), cudaMemcpyHostToDevice, st);
    };
    upload(&b->d_items, host);
    for (int k = 0; k < LISTS; ++k) upload(&b->d_units[k], units[k]);
    upload(&b->d_sums_fwd, sums_f);
    upload(&b->d_sums_bwd, sums_b);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_counters, LISTS * sizeof(int));
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        set_error("fmm_batch_create", e);
        fmm_batch_destroy(b);
        return e == cudaErrorMemoryAllocation ? FMM_ENOMEM : FMM_ECUDA;
    }
    if (dtype == FMM_BF16) {
        b->grid[0] = grid_for((const void *)batch_kernel<bf16_t, 0>, 256);
        b->grid[1] = grid_for((const void *)batch_kernel<bf16_t, 1>, 256);
        b->grid[2] = grid_for((const void *)ring_batch_kernel<M_FUSED, bf16_t>, 32);
        b->grid[3] = grid_for((const void *)ring_batch_kernel<M_BWD_ROW, bf16_t>, 32);
        b->grid[4] = grid_for((const void *)ring_batch_kernel<M_BWD_COL, bf16_t>, 32);
    } else {
        b->grid[0] = grid_for((const void *)batch_kernel<float, 0>, 256);
        b->grid[1] = grid_for((const void *)batch_kernel<float, 1>, 256);
        b->grid[3] = grid_for((const void *)ring_batch_kernel<M_BWD_ROW, float>, 32);
    }
    *batch = b;
    return FMM_OK;
}

// One phase: the units of the ring kernels, those of the team kernel, and the
// sums of the split rows.
static int run_phase(const fmm_batch *b, int phase, fmm_stream stream, const char *name)
{
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(b->d_counters, 0, LISTS * sizeof(int), st);
    auto run = [&](auto *kernel, int list, int threads) {
        if (e != cudaSuccess || b->n_units[list] == 0)
            return;
        kernel<<<b->grid[list], threads, 0, st>>>(b->d_items, b->d_units[list], b->n_units[list],
                                                  b->d_counters + list);
        e = cudaGetLastError();
    };
    const bool bf16 = b->dtype == FMM_BF16;
    if (phase == 0) {
        run(ring_batch_kernel<M_FUSED, bf16_t>, 2, 32);
        run(bf16 ? batch_kernel<bf16_t, 0> : batch_kernel<float, 0>, 0, 256);
    } else {
        run(bf16 ? ring_batch_kernel<M_BWD_ROW, bf16_t> : ring_batch_kernel<M_BWD_ROW, float>, 3, 32);
        run(ring_batch_kernel<M_BWD_COL, bf16_t>, 4, 32);
        run(bf16 ? batch_kernel<bf16_t, 1> : batch_kernel<float, 1>, 1, 256);
    }
    const int n_sums = phase ? b->n_sums_bwd : b->n_sums_fwd;
    if (e == cudaSuccess && n_sums > 0) {
        batch_sum_kernel<<<(n_sums + 3) / 4, 128, 0, st>>>(phase ? b->d_sums_bwd : b->d_sums_fwd,
                                                          n_sums);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error(name, e);
        return FMM_ECUDA;
    }
    return FMM_OK;
}

int fmm_batch_forward(const fmm_batch *b, fmm_stream stream)
{
    if (!b) {
        set_error_msg("batch is NULL");
        return FMM_EINVAL;
    }
    return run_phase(b, 0, stream, "fmm_batch_forward");
}

int fmm_batch_backward(const fmm_batch *b, fmm_stream stream)
{
    if (!b) {
        set_error_msg("batch is NULL");
        return FMM_EINVAL;
    }
    if (!b->has_bwd) {
        set_error_msg("batch built without G and gradient outputs (or without S^T)");
        return FMM_EUNSUPPORTED;
    }
    return run_phase(b, 1, stream, "fmm_batch_backward");
}

int fmm_batch_destroy(fmm_batch *b)
{
    if (!b)
        return FMM_OK;
    cudaDeviceSynchronize();
    cudaFree(b->d_items);
    for (int4 *u : b->d_units) cudaFree(u);
    cudaFree(b->d_counters);
    cudaFree(b->d_partials);
    cudaFree(b->d_sums_fwd);
    cudaFree(b->d_sums_bwd);
    delete b;
    return FMM_OK;
}

}  // extern "C"
