// Row pass for launches whose time is their longest rows: a whole warp per
// long row (or chunk), one lane group per row for the others, in one launch.
//
// With one lane group per row a team takes two nonzeros per dependent step of
// about 0.37 us (a gather from L2 and its use), so a row of 256 nonzeros takes
// 47 us however small the matrix is.  Here the first n_wide work items (they
// are in order of length) get a warp each:
//   * roles whose order of sums is free (bfloat16, SDDMM, the adjoints): the
//     lane groups of the warp take the nonzeros in turn, U each, and sum their
//     partial rows at the end;
//   * float32 FusedMM and SpMM keep the team kernel's order, bit for bit (see
//     fmm_flex.cuh): the groups compute the dot products of the next eight
//     nonzeros at once, in the team kernel's lane layout; then every lane,
//     owning r / 32 columns, adds the eight rows one after the other, reading
//     them a second time (from L1).  SpMM has only the second part.
// The other items run the team kernel's default layout in the remaining blocks.
// When the rule takes it, and what it measured, stands at wide_items in
// fmm_api.cu.
#pragma once

#include "fmm_flex.cuh"

namespace fmm {

template <typename T, int R>
constexpr int team_vpl()   // 8 elements per lane
{
    return sizeof(T) == 4 && R * 4 / 16 <= 32 ? 2 * base_vpl<T, R>() : base_vpl<T, R>();
}

// C floats of a row from a 4 C-byte-aligned address.
template <int C>
__device__ __forceinline__ void load_cols(const float *p, float (&f)[C])
{
#pragma unroll
    for (int q = 0; q < C / 4; ++q) {
        const float4 x = __ldg(reinterpret_cast<const float4 *>(p) + q);
        f[4 * q] = x.x; f[4 * q + 1] = x.y; f[4 * q + 2] = x.z; f[4 * q + 3] = x.w;
    }
    if constexpr (C == 2) {
        const float2 x = __ldg(reinterpret_cast<const float2 *>(p));
        f[0] = x.x; f[1] = x.y;
    }
    if constexpr (C == 1)
        f[0] = __ldg(p);
}

// Float32 FusedMM or SpMM of one item by a warp, in the team kernel's order.
template <int MODE, int R>
__device__ __forceinline__ void wide_ordered(const PassArgs &a, long long item, bool active)
{
    constexpr int Q = 8;                    // nonzeros per step
    constexpr int G = R / 8, NG = 32 / G;   // lanes per dot product, dot products at once
    constexpr int U = Q / NG;
    constexpr int C = R / 32;               // columns per lane in the sums
    const int lane = threadIdx.x & 31, lig = lane & (G - 1), grp = lane / G;
    int row = 0, beg = 0, end = 0, slot = -1;
    if (active)
        active = pass_item<false>(a, item, row, beg, end, slot);
    const float *L = static_cast<const float *>(a.L), *Y = static_cast<const float *>(a.Y);
    float l[8], acc[C] = {};
#pragma unroll
    for (int e = 0; e < 8; ++e) l[e] = 0.f;
    if (MODE == M_FUSED && end > beg) {
        const float *p = L + (size_t)row * R + 4 * lig;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const float4 x = __ldcs(reinterpret_cast<const float4 *>(p + 4 * G * v));
            l[4 * v] = x.x; l[4 * v + 1] = x.y; l[4 * v + 2] = x.z; l[4 * v + 3] = x.w;
        }
    }
    const unsigned n = (unsigned)(end - beg);   // uniform in the warp
    // lane q < Q holds the index and value of the step's nonzero q
    int j = 0;
    float s = 0.f;
    auto fetch = [&](unsigned k) {
        if (lane < Q && k + lane < n) {
            const int p = beg + (int)(k + lane);
            j = __ldg(a.col_idx + p);
            const int sp = (a.perm && !a.s_direct) ? __ldg(a.perm + p) : p;
            s = a.s ? __ldg(a.s + (a.s_direct ? p : sp)) : 1.f;
        }
    };
    fetch(0);
    for (unsigned k = 0; k < n; k += Q) {
        // positions past the end repeat earlier indices: loaded, not used
        int jq[Q];
        float sq[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            jq[q] = __shfl_sync(0xffffffffu, j, q);
            sq[q] = __shfl_sync(0xffffffffu, s, q);
        }
        float y[U][8];
        if constexpr (MODE == M_FUSED) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                // nonzero u NG + grp (a shuffle: grp is not a constant)
                const int jj = __shfl_sync(0xffffffffu, j, u * NG + grp);
                const float *p = Y + (size_t)jj * R + 4 * lig;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const float4 x = __ldg(reinterpret_cast<const float4 *>(p + 4 * G * v));
                    y[u][4 * v] = x.x; y[u][4 * v + 1] = x.y;
                    y[u][4 * v + 2] = x.z; y[u][4 * v + 3] = x.w;
                }
            }
        }
        float z[Q][C];
#pragma unroll
        for (int q = 0; q < Q; ++q)
            load_cols<C>(Y + (size_t)jq[q] * R + C * lane, z[q]);
        fetch(k + Q);
        float d[U];
        if constexpr (MODE == M_FUSED) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                d[u] = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) d[u] = fmaf(l[e], y[u][e], d[u]);
            }
            group_allreduce<G, U>(d);
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float c = sq[q];
            if constexpr (MODE == M_FUSED)
                c = c * __shfl_sync(0xffffffffu, d[q / NG], (q % NG) * G);
            if (k + q < n) {
#pragma unroll
                for (int t = 0; t < C; ++t) acc[t] = fmaf(c, z[q][t], acc[t]);
            }
        }
    }
    if (!active)
        return;
    float *dst = slot >= 0 ? a.partials + (size_t)slot * R
                           : (a.out ? a.out + (size_t)row * R : nullptr);
    if (!dst)
        return;
    const bool add = a.accumulate && slot < 0;
    dst += C * lane;
    if constexpr (C >= 4) {
        const Loader ld;
#pragma unroll
        for (int t = 0; t < C; t += 4)
            out_store4(ld, dst + t, make_float4(acc[t], acc[t + 1], acc[t + 2], acc[t + 3]), add);
    } else {
#pragma unroll
        for (int t = 0; t < C; ++t) dst[t] = add ? dst[t] + acc[t] : acc[t];
    }
}

template <int MODE, typename T, int R>
__device__ __forceinline__ void wide_item(const PassArgs &a, long long item, bool active)
{
    if constexpr (flex_ordered<MODE, T>()) {
        wide_ordered<MODE, R>(a, item, active);
    } else {
        // eight nonzeros or more in flight per warp
        constexpr int G = R / 8, NG = 32 / G, EPV = Elem<T>::PER16;
        constexpr int U = MODE == M_BWD_COL ? 2 : NG >= 4 ? 2 : 4;
        flex_item<MODE, T, 16, 8, U, false, false>(a, item, active, FlexShape{G, NG, R / EPV});
    }
}

constexpr int kWideBlock = 64;

template <int MODE, typename T, int R>
__global__ void __launch_bounds__(kWideBlock) wide_pass_kernel(const PassArgs a, int n_wide,
                                                              int wide_blocks)
{
    constexpr int V = team_vpl<T, R>();
    constexpr int TEAM = TeamShape<T, R, V, 1>::TEAM;
    if ((int)blockIdx.x < wide_blocks) {
        const long long item = (long long)blockIdx.x * (kWideBlock / 32) + (threadIdx.x >> 5);
        wide_item<MODE, T, R>(a, item, item < n_wide);
    } else {
        const long long gid =
            n_wide + ((long long)(blockIdx.x - wide_blocks) * kWideBlock + threadIdx.x) / TEAM;
        team_pass_body<MODE, T, R, V, 1, 2>(a, gid, gid < (long long)a.n_chunks + a.n_light);
    }
}

template <int MODE, typename T, int R>
cudaError_t launch_wide_width(const PassArgs &a, int n_wide, cudaStream_t st)
{
    constexpr int TEAM = TeamShape<T, R, team_vpl<T, R>(), 1>::TEAM;
    const long long rest = (long long)a.n_chunks + a.n_light - n_wide;
    const int wide_blocks = (n_wide + kWideBlock / 32 - 1) / (kWideBlock / 32);
    const long long blocks = wide_blocks + (rest * TEAM + kWideBlock - 1) / kWideBlock;
    wide_pass_kernel<MODE, T, R><<<(unsigned)blocks, kWideBlock, 0, st>>>(a, n_wide, wide_blocks);
    return cudaGetLastError();
}

template <typename T, int R>
cudaError_t dispatch_wide(int mode, const PassArgs &a, int n_wide, cudaStream_t st)
{
    switch (mode) {
    case M_FUSED: return launch_wide_width<M_FUSED, T, R>(a, n_wide, st);
    case M_SDDMM: return launch_wide_width<M_SDDMM, T, R>(a, n_wide, st);
    case M_SPMM: return launch_wide_width<M_SPMM, T, R>(a, n_wide, st);
    case M_BWD_ROW: return launch_wide_width<M_BWD_ROW, T, R>(a, n_wide, st);
    case M_BWD_COL: return launch_wide_width<M_BWD_COL, T, R>(a, n_wide, st);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_wide_typed(int mode, const PassArgs &a, int n_wide, cudaStream_t st)
{
    switch (a.r) {
    case 32: return dispatch_wide<T, 32>(mode, a, n_wide, st);
    case 64: return dispatch_wide<T, 64>(mode, a, n_wide, st);
    case 128: return dispatch_wide<T, 128>(mode, a, n_wide, st);
    case 256: return dispatch_wide<T, 256>(mode, a, n_wide, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fmm
