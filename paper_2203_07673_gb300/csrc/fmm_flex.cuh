// Row pass for any width and alignment, and for passes too small to fill the
// GPU with one lane group per row.
//
// The layouts of fmm_rows.cuh fix the row width, the lanes per row and the
// lane groups per row at compile time.  Here only the loads are fixed: a row
// of r elements is cut into vectors of VB bytes (the widest that divides the
// row and that every operand is aligned to), a lane holds E elements of it
// (E / EPV vectors, lane l the vectors l, l + G, ...; vectors past the row
// are zeros that are never loaded), and the G lanes of a group and the
// groups of a team are launch parameters.  The NG groups of a team take the
// nonzeros of their row or chunk in turn and sum their partial rows at the
// end in a fixed xor order.
//
// What bounds it: the gathers (L2 or HBM), as in the other passes; with the
// output row in registers each gathered row is read once.  Column indices
// and values of the next batch are loaded while the current one is used
// (every lane of a group reads the same word: one request per group).
// 8 elements per lane up to r = 256, as the team kernel's default layout (the
// light register footprint keeps more rows in flight), 12 up to 384, 16 up to
// 512; the roles that keep an order (below) as few as cover the row, since a
// vector step costs the same whether it holds elements or not (Erdos-Renyi,
// 60000 rows of 16, r = 25, float32, FusedMM: 149 us with 8 steps, 55 with 1).
//
// Measured on GB300 against the generic kernel, which it replaces for r <=
// 512 (us, Erdos-Renyi as above / Zipf rows, 60000 of 24): float32, r = 100:
// FusedMM 215 -> 43 / 399 -> 108, SDDMM 124 -> 43 / 247 -> 70, SpMM 136 -> 29 /
// 304 -> 79, adjoint over S 249 -> 67 / 488 -> 115, over S^T 260 -> 81 /
// 381 -> 112; r = 201: FusedMM 253 -> 97 / 516 -> 169, SDDMM 131 -> 91 /
// 251 -> 157, SpMM 211 -> 77 / 524 -> 134; bfloat16, r = 201: FusedMM 243 -> 161 /
// 504 -> 263, SDDMM 133 -> 120 / 232 -> 197, SpMM 183 -> 136 / 435 -> 229.
#pragma once

#include "fmm_rows.cuh"

namespace fmm {

struct FlexShape {
    int g;        // lanes per group (power of two, <= 32)
    int ng;       // groups per team (power of two, g * ng <= 32)
    int nvec;     // vectors per row
};

// One vector of VB bytes of a row of T, widened to EPV floats.
template <typename T, int VB>
__device__ __forceinline__ void flex_load(const T *p, float *f, bool gather)
{
    if constexpr (VB == 16) {
        const uint4 *q = reinterpret_cast<const uint4 *>(p);
        const uint4 w = gather ? __ldg(q) : __ldcs(q);
        if constexpr (sizeof(T) == 2) {
            unpack_bf16x8(w, f);
        } else {
            f[0] = __uint_as_float(w.x); f[1] = __uint_as_float(w.y);
            f[2] = __uint_as_float(w.z); f[3] = __uint_as_float(w.w);
        }
    } else if constexpr (VB == 8) {
        const uint2 *q = reinterpret_cast<const uint2 *>(p);
        const uint2 w = gather ? __ldg(q) : __ldcs(q);
        if constexpr (sizeof(T) == 2) {
            f[0] = __uint_as_float(w.x << 16); f[1] = __uint_as_float(w.x & 0xffff0000u);
            f[2] = __uint_as_float(w.y << 16); f[3] = __uint_as_float(w.y & 0xffff0000u);
        } else {
            f[0] = __uint_as_float(w.x); f[1] = __uint_as_float(w.y);
        }
    } else if constexpr (VB == 4) {
        const uint32_t *q = reinterpret_cast<const uint32_t *>(p);
        const uint32_t w = gather ? __ldg(q) : __ldcs(q);
        if constexpr (sizeof(T) == 2) {
            f[0] = __uint_as_float(w << 16); f[1] = __uint_as_float(w & 0xffff0000u);
        } else {
            f[0] = __uint_as_float(w);
        }
    } else {
        static_assert(sizeof(T) == 2, "two-byte vectors are bfloat16 elements");
        f[0] = widen<T>(gather ? __ldg(p) : __ldcs(p));
    }
}

// EPV floats from or to an address aligned to min(16, 4 EPV) bytes.
template <int EPV>
__device__ __forceinline__ void flex_load_f32(const float *p, float *f, bool gather)
{
    if constexpr (EPV % 4 == 0) {
#pragma unroll
        for (int q = 0; q < EPV / 4; ++q) {
            const float4 *a = reinterpret_cast<const float4 *>(p) + q;
            const float4 x = gather ? __ldg(a) : __ldcs(a);
            f[4 * q] = x.x; f[4 * q + 1] = x.y; f[4 * q + 2] = x.z; f[4 * q + 3] = x.w;
        }
    } else if constexpr (EPV == 2) {
        const float2 *a = reinterpret_cast<const float2 *>(p);
        const float2 x = gather ? __ldg(a) : __ldcs(a);
        f[0] = x.x; f[1] = x.y;
    } else {
        f[0] = gather ? __ldg(p) : __ldcs(p);
    }
}

template <int EPV>
__device__ __forceinline__ void flex_store_f32(float *p, const float *f, bool add)
{
    if constexpr (EPV % 4 == 0) {
        const Loader ld;
#pragma unroll
        for (int q = 0; q < EPV / 4; ++q)
            out_store4(ld, p + 4 * q, make_float4(f[4 * q], f[4 * q + 1], f[4 * q + 2], f[4 * q + 3]),
                       add);
    } else if constexpr (EPV == 2) {
        float2 v = make_float2(f[0], f[1]);
        if (add) {
            const float2 o = __ldcs(reinterpret_cast<const float2 *>(p));
            v.x += o.x; v.y += o.y;
        }
        __stcs(reinterpret_cast<float2 *>(p), v);
    } else {
        __stcs(p, add ? f[0] + __ldcs(p) : f[0]);
    }
}

// EPV floats as bfloat16 to an address aligned to 2 EPV bytes.
template <int EPV>
__device__ __forceinline__ void flex_store_bf16(uint16_t *p, const float *f)
{
    if constexpr (EPV == 8) {
        store_bf16x8(p, f);
    } else if constexpr (EPV == 4) {
        __stcs(reinterpret_cast<uint2 *>(p), make_uint2(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3])));
    } else if constexpr (EPV == 2) {
        __stcs(reinterpret_cast<uint32_t *>(p), pack_bf16x2(f[0], f[1]));
    } else {
        *p = (uint16_t)pack_bf16x2(f[0], 0.f);
    }
}

// Whether a role adds in the order of the generic kernel: float32 FusedMM and
// SpMM, whose results an iteration may amplify (the conjugate gradients of
// ALS past their convergence), are the same bits as the generic kernel's.
// That fixes the lanes of a group (32 / EPV, so that element e of vector v of
// lane l is element 32 v + EPV l + e: position EPV l + e of the generic
// kernel's warp, step v), one group per row, and the order of the dot product
// below.
template <int MODE, typename T>
constexpr bool flex_ordered() { return sizeof(T) == 4 && (MODE == M_FUSED || MODE == M_SPMM); }

// Sum over the 32 / EPV lanes of a group and the EPV elements of each, in the
// order of a 32-lane xor butterfly over positions EPV l + e (offsets 16, 8,
// 4, 2, 1).  The first offsets cross lanes, the last ones elements; a lane
// keeps half of its elements at each of the first log2(EPV) offsets, so the
// elements' offsets become one shuffle each at the end.
template <int EPV>
__device__ __forceinline__ float ordered_sum(const float (&d)[EPV], int lig)
{
    constexpr unsigned ALL = 0xffffffffu;
    if constexpr (EPV == 4) {
        const bool b2 = lig & 4, b1 = lig & 2;
        const float s0 = __shfl_xor_sync(ALL, b2 ? d[0] : d[2], 4);
        const float s1 = __shfl_xor_sync(ALL, b2 ? d[1] : d[3], 4);
        const float k0 = (b2 ? d[2] : d[0]) + s0, k1 = (b2 ? d[3] : d[1]) + s1;   // 16
        float m = (b1 ? k1 : k0) + __shfl_xor_sync(ALL, b1 ? k0 : k1, 2);         // 8
        m += __shfl_xor_sync(ALL, m, 1);                                          // 4
        m += __shfl_xor_sync(ALL, m, 4);                                          // 2
        m += __shfl_xor_sync(ALL, m, 2);                                          // 1
        return m;
    } else if constexpr (EPV == 2) {
        const bool b3 = lig & 8;
        float m = (b3 ? d[1] : d[0]) + __shfl_xor_sync(ALL, b3 ? d[0] : d[1], 8);   // 16
        m += __shfl_xor_sync(ALL, m, 4);                                            // 8
        m += __shfl_xor_sync(ALL, m, 2);                                            // 4
        m += __shfl_xor_sync(ALL, m, 1);                                            // 2
        m += __shfl_xor_sync(ALL, m, 8);                                            // 1
        return m;
    } else {
        return warp_allreduce(d[0]);
    }
}

// Accumulates into acc the nonzeros beg + first, beg + first + step, ... of
// [beg, end): the share of one group of g lanes (lig = lane within it).
// Every lane of the warp must call it.  U: nonzeros per batch; ORD: in the
// generic kernel's order.
template <int MODE, typename T, int VB, int E, int U, bool ORD, bool CHECK>
__device__ __forceinline__ void flex_range(const PassArgs &a, int row, int beg, int end, int first,
                                           int step, int g, int lig, int nvec, float (&acc)[E])
{
    constexpr int EPV = VB / (int)sizeof(T), VPL = E / EPV;
    constexpr bool HAS_L = MODE != M_SPMM;
    constexpr bool TWO = MODE == M_BWD_ROW || MODE == M_BWD_COL;
    constexpr bool NZ = MODE == M_SDDMM || MODE == M_BWD_ROW;
    constexpr int ND = TWO ? 2 * U : U;
    static_assert(E % EPV == 0, "whole vectors per lane");

    const int r = a.r;
    const T *L = static_cast<const T *>(a.L);
    const T *Y = static_cast<const T *>(a.Y);
    // lane's first element; vector v of the lane starts at k0 + v * vs
    const int k0 = lig * EPV, vs = g * EPV;
    const int mine = lig < nvec ? (nvec - lig + g - 1) / g : 0;   // vectors of this lane

    float lrow[E], hrow[MODE == M_BWD_ROW ? E : 1];
#pragma unroll
    for (int e = 0; e < E; ++e) { lrow[e] = 0.f; acc[e] = 0.f; }
#pragma unroll
    for (int e = 0; e < (MODE == M_BWD_ROW ? E : 1); ++e) hrow[e] = 0.f;
    if (HAS_L && end > beg) {
#pragma unroll
        for (int v = 0; v < VPL; ++v)
            if (v < mine) {
                flex_load<T, VB>(L + (size_t)row * r + k0 + v * vs, &lrow[v * EPV], false);
                if constexpr (MODE == M_BWD_ROW)
                    flex_load_f32<EPV>(a.H + (size_t)row * r + k0 + v * vs, &hrow[v * EPV], false);
            }
    }

    // positions relative to beg, unsigned: past the end they cannot wrap
    const unsigned n = (unsigned)(end - beg), span = (unsigned)(U * step);
    const unsigned iters = n > (unsigned)first ? (n - first + span - 1) / span : 0;
    const unsigned witers = __reduce_max_sync(0xffffffffu, iters);
    unsigned q = first;
    int jn[U], sin_[U];
    float svn[U];
    auto fetch = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            jn[u] = -1; sin_[u] = 0; svn[u] = 0.f;
            if (q + u * step < n) {
                const int pp = beg + (int)(q + u * step);
                jn[u] = pass_col<CHECK>(a, pp);
                sin_[u] = (a.perm && (NZ || !a.s_direct)) ? __ldg(a.perm + pp) : pp;
                svn[u] = a.s ? __ldg(a.s + (a.s_direct ? pp : sin_[u])) : 1.f;
            }
        }
    };
    fetch();
    for (unsigned it = 0; it < witers; ++it) {
        int jj[U], sidx[U];
        float sv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) { jj[u] = jn[u]; sidx[u] = sin_[u]; sv[u] = svn[u]; }
        float y[U][E], h[MODE == M_BWD_COL ? U : 1][E];
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                y[u][e] = 0.f;
                if constexpr (MODE == M_BWD_COL) h[u][e] = 0.f;
            }
            if (jj[u] >= 0) {
                const T *yp = Y + (size_t)jj[u] * r + k0;
#pragma unroll
                for (int v = 0; v < VPL; ++v)
                    if (v < mine)
                        flex_load<T, VB>(yp + v * vs, &y[u][v * EPV], true);
                if constexpr (MODE == M_BWD_COL) {
                    const float *hp = a.H + (size_t)jj[u] * r + k0;
#pragma unroll
                    for (int v = 0; v < VPL; ++v)
                        if (v < mine)
                            flex_load_f32<EPV>(hp + v * vs, &h[u][v * EPV], true);
                }
            }
        }
        q += span;
        fetch();
        if constexpr (MODE == M_SPMM) {
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (jj[u] >= 0)
                        acc[e] = fmaf(sv[u], y[u][e], acc[e]);
            continue;
        }
        float d[ND];
        if constexpr (ORD) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float de[EPV] = {};
#pragma unroll
                for (int v = 0; v < VPL; ++v)
#pragma unroll
                    for (int e = 0; e < EPV; ++e)
                        de[e] = fmaf(lrow[v * EPV + e], y[u][v * EPV + e], de[e]);
                d[u] = ordered_sum<EPV>(de, lig);
            }
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float t = 0.f;
#pragma unroll
                for (int e = 0; e < E; ++e) t = fmaf(lrow[e], y[u][e], t);
                d[u] = t;
                if constexpr (TWO) {
                    float w = 0.f;
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        w = MODE == M_BWD_ROW ? fmaf(hrow[MODE == M_BWD_ROW ? e : 0], y[u][e], w)
                                              : fmaf(h[MODE == M_BWD_COL ? u : 0][e], lrow[e], w);
                    d[U + u] = w;
                }
            }
            for (int off = g >> 1; off > 0; off >>= 1) {
#pragma unroll
                for (int i = 0; i < ND; ++i)
                    d[i] += __shfl_xor_sync(0xffffffffu, d[i], off);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (jj[u] < 0)
                continue;
            if constexpr (MODE == M_FUSED) {
                const float c = sv[u] * d[u];
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] = fmaf(c, y[u][e], acc[e]);
            } else if constexpr (MODE == M_SDDMM) {
                if (lig == 0)
                    nz_store<MODE>(a, sidx[u], sv[u] * d[u]);
            } else if constexpr (MODE == M_BWD_ROW) {
                if (lig == 0 && a.nzout)
                    a.nzout[sidx[u]] = d[u] * d[U + u];
                const float c = sv[u] * d[U + u];
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] = fmaf(c, y[u][e], acc[e]);
            } else if constexpr (MODE == M_BWD_COL) {
                const float c1 = sv[u] * d[u], c2 = sv[u] * d[U + u];
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] = fmaf(c1, h[u][e], fmaf(c2, y[u][e], acc[e]));
            }
        }
    }
}

// Work item `item` by a team of sh.g x sh.ng lanes.
template <int MODE, typename T, int VB, int E, int U, bool ORD, bool CHECK>
__device__ __forceinline__ void flex_item(const PassArgs &a, long long item, bool active,
                                          const FlexShape &sh)
{
    constexpr int EPV = VB / (int)sizeof(T), VPL = E / EPV;
    const int team = sh.g * sh.ng;
    const int lane = threadIdx.x & 31;
    const int lig = lane & (sh.g - 1);
    const int grp = (lane & (team - 1)) / sh.g;
    int row = 0, beg = 0, end = 0, slot = -1;
    if (active)
        active = pass_item<CHECK>(a, item, row, beg, end, slot);
    float acc[E];
    flex_range<MODE, T, VB, E, U, ORD, CHECK>(a, row, beg, end, grp, sh.ng, sh.g, lig, sh.nvec, acc);
    if constexpr (MODE != M_SDDMM) {
        for (int off = sh.g; off < team; off <<= 1) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], off);
        }
        if (!active || grp != 0)
            return;
        float *dst = slot >= 0 ? a.partials + (size_t)slot * a.r
                               : (a.out ? a.out + (size_t)row * a.r : nullptr);
        if constexpr (sizeof(T) == 2 && (MODE == M_BWD_ROW || MODE == M_BWD_COL)) {
            if (a.out16 && slot < 0) {
#pragma unroll
                for (int v = 0; v < VPL; ++v)
                    if (v * sh.g + lig < sh.nvec)
                        flex_store_bf16<EPV>(a.out16 + (size_t)row * a.r + (v * sh.g + lig) * EPV,
                                             &acc[v * EPV]);
                return;
            }
        }
        if (!dst)
            return;
#pragma unroll
        for (int v = 0; v < VPL; ++v)
            if (v * sh.g + lig < sh.nvec)
                flex_store_f32<EPV>(dst + (v * sh.g + lig) * EPV, &acc[v * EPV],
                                    a.accumulate && slot < 0);
    }
}

// Blocks of two warps, as the team kernel's; register caps of 64 per thread
// in the forward roles, 72 in the pass over S, 80 in the pass over S^T (the
// narrow vectors of the adjoints spill up to 40 bytes).
constexpr int kFlexBlock = 64;

template <int MODE, int E>
constexpr int flex_min_blocks()
{
    return E > 12 ? 8 : E > 8 ? (MODE == M_BWD_COL ? 8 : 10)
         : MODE == M_BWD_COL ? 12 : MODE == M_BWD_ROW ? 14 : 16;
}

// Roles whose order is free give the first n_wide items (chunks and rows of 64
// nonzeros or more; the items are in order of length) all lane groups of a
// warp; the other items take sh (Zipf rows, 60000 of 24, bfloat16, r = 25:
// FusedMM 160 -> 73 us, SpMM 180 -> 79: a chunk of 256 nonzeros on one group of
// four lanes was the pass).  G > 0: the lanes of a group as a constant, so the
// vectors of a row lie at constant offsets (Erdos-Renyi, 60000 rows of 16,
// r = 201: float32 FusedMM 156 -> 97, SDDMM 153 -> 91, bfloat16 adjoint over S
// 270 -> 204).
template <int MODE, typename T, int VB, int E, int G, bool ORD, bool CHECK>
__global__ void __launch_bounds__(kFlexBlock, flex_min_blocks<MODE, E>())
    flex_pass_kernel(const PassArgs a, FlexShape sh, int n_wide, int wide_blocks)
{
    const long long total = (long long)a.n_chunks + a.n_light;
    long long item = ((long long)blockIdx.x - wide_blocks) * blockDim.x + threadIdx.x;
    if constexpr (G > 0)
        sh.g = G;
    if constexpr (ORD || G == 32)
        sh.ng = 1;
    if (!ORD && G < 32 && (int)blockIdx.x < wide_blocks) {
        sh.ng = 32 / sh.g;
        item = (long long)blockIdx.x * (kFlexBlock / 32) + (threadIdx.x >> 5);
        if (item >= n_wide)
            item = total;
    } else {
        item = n_wide + item / (sh.g * sh.ng);
    }
    flex_item<MODE, T, VB, E, (ORD && E <= 4 ? 4 : E <= 8 ? 2 : 1), ORD, CHECK>(a, item,
                                                                               item < total, sh);
}

template <int MODE, typename T, int VB, int E, int G, bool ORD, bool CHECK>
cudaError_t launch_flex_shape(const PassArgs &a, int ng, cudaStream_t st)
{
    constexpr int EPV = VB / (int)sizeof(T), WB = kFlexBlock / 32;
    FlexShape sh;
    sh.nvec = a.r / EPV;
    sh.g = G > 0 ? G : flex_lanes(a.r);
    sh.ng = 1;
    while (!ORD && sh.ng < ng && sh.g * sh.ng < 32) sh.ng *= 2;
    int n_wide = 0;
    if (!ORD && a.bucket_start && sh.g * sh.ng < 32)
        n_wide = a.n_chunks + a.bucket_start[length_key(64, INT32_MAX) + 1] - a.bucket_start[1];
    const int wide_blocks = (n_wide + WB - 1) / WB;
    const long long rest = (long long)a.n_chunks + a.n_light - n_wide;
    const long long blocks = wide_blocks + (rest * sh.g * sh.ng + kFlexBlock - 1) / kFlexBlock;
    flex_pass_kernel<MODE, T, VB, E, G, ORD, CHECK>
        <<<(unsigned)blocks, kFlexBlock, 0, st>>>(a, sh, n_wide, wide_blocks);
    return cudaGetLastError();
}

// vb: bytes per vector (a power of two up to 16, a multiple of the element
// size, dividing the row and the alignment of every operand).  Roles that
// keep the generic kernel's order hold 32 elements of a row per vector step,
// so a lane's E elements cover r <= 32 E / EPV: narrower vectors for wider
// rows.
template <int MODE, typename T, bool ORD = flex_ordered<MODE, T>(), bool CHECK = false>
cudaError_t dispatch_flex(const PassArgs &a, int vb, int ng, cudaStream_t st)
{
    if constexpr (ORD) {
        while (vb > 4 && a.r > 32 * 16 / (vb / 4)) vb /= 2;
#define FMM_FLEX(VB, E)                                                           \
    if (vb == VB && a.r <= 32 * E / (VB / 4))                                     \
        return launch_flex_shape<MODE, T, VB, E, 128 / VB, ORD, CHECK>(a, ng, st);
        FMM_FLEX(16, 4) FMM_FLEX(16, 8) FMM_FLEX(16, 16)
        FMM_FLEX(8, 2) FMM_FLEX(8, 4) FMM_FLEX(8, 8) FMM_FLEX(8, 16)
        FMM_FLEX(4, 1) FMM_FLEX(4, 2) FMM_FLEX(4, 4) FMM_FLEX(4, 8) FMM_FLEX(4, 16)
#undef FMM_FLEX
        return cudaErrorInvalidValue;
    }
    // 12 elements up to r = 384 where vectors allow it (Erdos-Renyi, 60000 rows
    // of 16, r = 300, bfloat16, FusedMM: 199 us with 16 elements, 166 with 12)
#define FMM_FLEX(VB)                                                              \
    if (vb == VB) {                                                               \
        if (a.r <= 32)                                                            \
            return launch_flex_shape<MODE, T, VB, 8, 0, ORD, CHECK>(a, ng, st);   \
        if (a.r <= 64)                                                            \
            return launch_flex_shape<MODE, T, VB, 8, 8, ORD, CHECK>(a, ng, st);   \
        if (a.r <= 128)                                                           \
            return launch_flex_shape<MODE, T, VB, 8, 16, ORD, CHECK>(a, ng, st);  \
        if (a.r <= 256)                                                           \
            return launch_flex_shape<MODE, T, VB, 8, 32, ORD, CHECK>(a, ng, st);  \
        if constexpr (VB / sizeof(T) <= 4)                                        \
            if (a.r <= 384)                                                       \
                return launch_flex_shape<MODE, T, VB, 12, 32, ORD, CHECK>(a, ng, st); \
        return launch_flex_shape<MODE, T, VB, 16, 32, ORD, CHECK>(a, ng, st);     \
    }
    FMM_FLEX(16)
    FMM_FLEX(8)
    FMM_FLEX(4)
    if constexpr (sizeof(T) == 2) {
        FMM_FLEX(2)
    }
#undef FMM_FLEX
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_flex_typed(int mode, const PassArgs &a, int vb, int ng, cudaStream_t st)
{
    if ((long long)a.n_chunks + a.n_light == 0)
        return cudaSuccess;
    switch (mode) {
    case M_FUSED: return dispatch_flex<M_FUSED, T>(a, vb, ng, st);
    case M_SDDMM: return dispatch_flex<M_SDDMM, T>(a, vb, ng, st);
    case M_SPMM: return dispatch_flex<M_SPMM, T>(a, vb, ng, st);
    case M_BWD_ROW: return dispatch_flex<M_BWD_ROW, T>(a, vb, ng, st);
    case M_BWD_COL: return dispatch_flex<M_BWD_COL, T>(a, vb, ng, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fmm
