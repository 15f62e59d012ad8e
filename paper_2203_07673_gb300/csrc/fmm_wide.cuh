// Row pass for launches whose time is their longest rows: a whole warp per
// long row (or chunk), one lane group per row for the others, in one launch.
//
// With one lane group per row a team takes two nonzeros per dependent step of
// about 0.37 us (a gather from L2 and its use), so a row of 256 nonzeros takes
// 47 us however small the matrix is.  Here the first n_wide work items (they
// are in order of length) get a warp each.
//
// The order of sums is that of the pass a role runs otherwise (the team kernel,
// or the register ring for bfloat16 FusedMM and adjoint over S), so neither the
// choice of this pass nor a batch (fmm_batch.cu), which has no such choice,
// changes a bit: the groups of the warp compute the dot products of the next
// eight nonzeros or more at once, in the lane layout of that pass; then every
// lane, owning r / 32 columns, adds their rows one after the other, reading them
// a second time (from L1).  SpMM has only the second part.  SDDMM has no sums
// over nonzeros, and bfloat16 SpMM is in no batch: they run as the
// flexible-width pass does, the groups taking the nonzeros in turn.
// The other items run the team kernel's default layout, or the ring, in the
// remaining blocks.
// When the rule takes it, and what it measured, stands at wide_items in
// fmm_api.cu.
#pragma once

#include "fmm_flex.cuh"
#include "fmm_pipe.cuh"

namespace fmm {

template <typename T, int R>
constexpr int team_vpl()   // 8 elements per lane
{
    return sizeof(T) == 4 && R * 4 / 16 <= 32 ? 2 * base_vpl<T, R>() : base_vpl<T, R>();
}

// C elements of a row as floats, from an address aligned to them (to 16 bytes
// where they are more).
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

template <int C>
__device__ __forceinline__ void load_cols(const bf16_t *p, float (&f)[C])
{
    static_assert(C <= 4, "bfloat16 rows of r <= 128");
    flex_load<bf16_t, 2 * C>(p, f, true);
}

// Lane layout of the dot products: RING as pipe_pass_body with two words per
// lane (16 consecutive elements, even and odd ones summed apart), else as the
// team kernel with 8 elements per lane.
template <typename T, int R, bool RING>
struct WideLayout {
    static constexpr int E = RING ? 16 : 8;           // elements per lane
    static constexpr int G = R / E, NG = 32 / G;      // lanes per dot product, products at once
    static constexpr int EPV = Elem<T>::PER16, VPL = E / EPV;
    // first element of the lane's word v
    static __device__ __forceinline__ int at(int lig, int v)
    {
        return RING ? (lig * VPL + v) * EPV : (v * G + lig) * EPV;
    }
    static __device__ __forceinline__ void load(const T *row, int lig, float (&f)[E])
    {
#pragma unroll
        for (int v = 0; v < VPL; ++v)
            unpack16<T>(__ldg(reinterpret_cast<const uint4 *>(row + at(lig, v))), &f[v * EPV]);
    }
    static __device__ __forceinline__ void load_f32(const float *row, int lig, float (&f)[E])
    {
#pragma unroll
        for (int e = 0; e < E; e += 4) {
            const float4 x = __ldg(reinterpret_cast<const float4 *>(row + at(lig, e / EPV) + e % EPV));
            f[e] = x.x; f[e + 1] = x.y; f[e + 2] = x.z; f[e + 3] = x.w;
        }
    }
    // the lane's part of <x, y>
    static __device__ __forceinline__ float dot(const float (&x)[E], const float (&y)[E])
    {
        if constexpr (RING) {
            float even = 0.f, odd = 0.f;
#pragma unroll
            for (int e = 0; e < E; e += 2) {
                even = fmaf(x[e], y[e], even);
                odd = fmaf(x[e + 1], y[e + 1], odd);
            }
            return even + odd;
        } else {
            float t = 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e) t = fmaf(x[e], y[e], t);
            return t;
        }
    }
};

// One item by a warp, in the order of sums described above.  DEEP: twice the
// nonzeros per step in rows of r <= 64, for launches whose warps are few (at
// most 16 per SM), where registers cost nothing (float32, r = 64, FusedMM, R-MAT
// of 2^12 vertices 18.4 -> 12.4 us, of 2^16 33 -> 38).
template <int MODE, typename T, int R, bool RING, bool DEEP>
__device__ __forceinline__ void wide_ordered(const PassArgs &a, long long item, bool active)
{
    using W = WideLayout<T, R, RING>;
    constexpr bool DOTS = MODE != M_SPMM, TWO = MODE == M_BWD_ROW || MODE == M_BWD_COL;
    constexpr int E = W::E, G = W::G, NG = W::NG;
    // nonzeros per step: as many as their rows have registers for
    constexpr int ROOM =
        (MODE == M_BWD_COL ? (R <= 64 ? 256 : 512) / R : 8) * (DEEP && R <= 64 ? 2 : 1);
    constexpr int U = NG >= ROOM ? 1 : ROOM / NG, Q = NG * U;
    constexpr int C = R / 32;               // columns per lane in the sums
    constexpr int ND = TWO ? 2 * U : U;
    const int lane = threadIdx.x & 31, lig = lane & (G - 1), grp = lane / G;
    int row = 0, beg = 0, end = 0, slot = -1;
    if (active)
        active = pass_item<false>(a, item, row, beg, end, slot);
    const T *L = static_cast<const T *>(a.L), *Y = static_cast<const T *>(a.Y);
    float l[E], lh[MODE == M_BWD_ROW ? E : 1], acc[C] = {};
    if (DOTS && end > beg) {   // uniform in the warp
        W::load(L + (size_t)row * R, lig, l);
        if constexpr (MODE == M_BWD_ROW)
            W::load_f32(a.H + (size_t)row * R, lig, lh);
    }
    const unsigned n = (unsigned)(end - beg);
    // lane q < Q holds the index, the value and the place in S of the step's
    // nonzero q
    int j = 0, si = 0;
    float s = 0.f;
    auto fetch = [&](unsigned k) {
        if (lane < Q && k + lane < n) {
            const int p = beg + (int)(k + lane);
            j = __ldg(a.col_idx + p);
            si = (a.perm && (MODE == M_BWD_ROW || !a.s_direct)) ? __ldg(a.perm + p) : p;
            s = a.s ? __ldg(a.s + (a.s_direct ? p : si)) : 1.f;
        }
    };
    fetch(0);
    for (unsigned k = 0; k < n; k += Q) {
        // positions past the end repeat earlier indices: loaded, not used
        int jq[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) jq[q] = __shfl_sync(0xffffffffu, j, q);
        // nonzero u NG + grp (a shuffle: grp is not a constant)
        float y[U][E], h[MODE == M_BWD_COL ? U : 1][E], su[U];
        int siu[U];
        const float sk = s;
        if constexpr (DOTS) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                su[u] = __shfl_sync(0xffffffffu, s, u * NG + grp);
                siu[u] = MODE == M_BWD_ROW ? __shfl_sync(0xffffffffu, si, u * NG + grp) : 0;
                const int jj = __shfl_sync(0xffffffffu, j, u * NG + grp);
                W::load(Y + (size_t)jj * R, lig, y[u]);
                if constexpr (MODE == M_BWD_COL)
                    W::load_f32(a.H + (size_t)jj * R, lig, h[u]);
            }
        }
        float z[Q][C], zh[MODE == M_BWD_COL ? Q : 1][C];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            load_cols<C>(Y + (size_t)jq[q] * R + C * lane, z[q]);
            if constexpr (MODE == M_BWD_COL)
                load_cols<C>(a.H + (size_t)jq[q] * R + C * lane, zh[q]);
        }
        fetch(k + Q);
        // coefficients of the rows: c of Y's, ch of H's
        float c[U], ch[MODE == M_BWD_COL ? U : 1];
        if constexpr (DOTS) {
            float d[ND];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                d[u] = W::dot(l, y[u]);
                if constexpr (MODE == M_BWD_ROW) d[U + u] = W::dot(lh, y[u]);
                if constexpr (MODE == M_BWD_COL) d[U + u] = W::dot(h[u], l);
            }
            group_allreduce<G, ND>(d);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                c[u] = su[u] * d[TWO ? U + u : u];
                if constexpr (MODE == M_BWD_COL) ch[u] = su[u] * d[u];
                if constexpr (MODE == M_BWD_ROW)
                    if (a.nzout && lig == 0 && k + u * NG + grp < n)
                        a.nzout[siu[u]] = d[u] * d[U + u];
            }
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float cq = DOTS ? __shfl_sync(0xffffffffu, c[q / NG], (q % NG) * G)
                                  : __shfl_sync(0xffffffffu, sk, q);
            float hq = 0.f;
            if constexpr (MODE == M_BWD_COL)
                hq = __shfl_sync(0xffffffffu, ch[q / NG], (q % NG) * G);
            if (k + q < n) {
#pragma unroll
                for (int t = 0; t < C; ++t) {
                    acc[t] = fmaf(cq, z[q][t], acc[t]);
                    if constexpr (MODE == M_BWD_COL) acc[t] = fmaf(hq, zh[q][t], acc[t]);
                }
            }
        }
    }
    if (!active)
        return;
    if constexpr (TWO && sizeof(T) == 2) {
        if (a.out16 && slot < 0) {
            flex_store_bf16<C>(a.out16 + (size_t)row * R + C * lane, acc);
            return;
        }
    }
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

template <int MODE, typename T, int R, bool RING, bool DEEP>
__device__ __forceinline__ void wide_item(const PassArgs &a, long long item, bool active)
{
    if constexpr (MODE != M_SDDMM && !(MODE == M_SPMM && sizeof(T) == 2)) {
        wide_ordered<MODE, T, R, RING, DEEP>(a, item, active);
    } else {
        // eight nonzeros or more in flight per warp
        constexpr int G = R / 8, NG = 32 / G, EPV = Elem<T>::PER16;
        flex_item<MODE, T, 16, 8, (NG >= 4 ? 2 : 4), false, false>(a, item, active,
                                                                   FlexShape{G, NG, R / EPV});
    }
}

constexpr int kWideBlock = 64;

// REST: there are items without a warp of their own (without them the kernel
// needs fewer registers: more of the short launches that give every row a warp
// are resident at once).
template <int MODE, typename T, int R, bool RING, bool REST, bool DEEP>
__global__ void __launch_bounds__(kWideBlock) wide_pass_kernel(const PassArgs a, int n_wide,
                                                              int wide_blocks)
{
    constexpr int V = RING ? 2 : team_vpl<T, R>();
    constexpr int TEAM = TeamShape<T, R, V, 1>::TEAM;
    if (!REST || (int)blockIdx.x < wide_blocks) {
        const long long item = (long long)blockIdx.x * (kWideBlock / 32) + (threadIdx.x >> 5);
        wide_item<MODE, T, R, RING, DEEP>(a, item, item < n_wide);
    } else {
        const long long gid =
            n_wide + ((long long)(blockIdx.x - wide_blocks) * kWideBlock + threadIdx.x) / TEAM;
        const bool active = gid < (long long)a.n_chunks + a.n_light;
        if constexpr (RING)
            pipe_pass_body<MODE, T, R, V, 1, 2, 1, false>(a, gid, active);
        else
            team_pass_body<MODE, T, R, V, 1, 2>(a, gid, active);
    }
}

template <int MODE, typename T, int R, bool RING>
cudaError_t launch_wide_width(const PassArgs &a, int n_wide, cudaStream_t st)
{
    constexpr int TEAM = TeamShape<T, R, RING ? 2 : team_vpl<T, R>(), 1>::TEAM;
    const long long rest = (long long)a.n_chunks + a.n_light - n_wide;
    const int wide_blocks = (n_wide + kWideBlock / 32 - 1) / (kWideBlock / 32);
    const long long blocks = wide_blocks + (rest * TEAM + kWideBlock - 1) / kWideBlock;
    const bool deep = n_wide <= 16 * sm_count();
    auto *kernel = rest > 0 ? (deep ? wide_pass_kernel<MODE, T, R, RING, true, true>
                                    : wide_pass_kernel<MODE, T, R, RING, true, false>)
                            : (deep ? wide_pass_kernel<MODE, T, R, RING, false, true>
                                    : wide_pass_kernel<MODE, T, R, RING, false, false>);
    kernel<<<(unsigned)blocks, kWideBlock, 0, st>>>(a, n_wide, wide_blocks);
    return cudaGetLastError();
}

// ring: whether the pass would otherwise run the register ring (bfloat16
// FusedMM and adjoint over S with 32-byte aligned gathered rows).
template <int MODE, typename T, int R>
cudaError_t launch_wide_mode(const PassArgs &a, int n_wide, bool ring, cudaStream_t st)
{
    if constexpr (wide_role(MODE, sizeof(T) == 2, R)) {
        if constexpr (sizeof(T) == 2 && (MODE == M_FUSED || MODE == M_BWD_ROW))
            if (ring)
                return launch_wide_width<MODE, T, R, true>(a, n_wide, st);
        return launch_wide_width<MODE, T, R, false>(a, n_wide, st);
    }
    return cudaErrorInvalidValue;
}

template <typename T, int R>
cudaError_t dispatch_wide(int mode, const PassArgs &a, int n_wide, bool ring, cudaStream_t st)
{
    switch (mode) {
    case M_FUSED: return launch_wide_mode<M_FUSED, T, R>(a, n_wide, ring, st);
    case M_SDDMM: return launch_wide_mode<M_SDDMM, T, R>(a, n_wide, ring, st);
    case M_SPMM: return launch_wide_mode<M_SPMM, T, R>(a, n_wide, ring, st);
    case M_BWD_ROW: return launch_wide_mode<M_BWD_ROW, T, R>(a, n_wide, ring, st);
    case M_BWD_COL: return launch_wide_mode<M_BWD_COL, T, R>(a, n_wide, ring, st);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_wide_typed(int mode, const PassArgs &a, int n_wide, bool ring, cudaStream_t st)
{
    switch (a.r) {
    case 32: return dispatch_wide<T, 32>(mode, a, n_wide, ring, st);
    case 64: return dispatch_wide<T, 64>(mode, a, n_wide, ring, st);
    case 128: return dispatch_wide<T, 128>(mode, a, n_wide, ring, st);
    case 256: return dispatch_wide<T, 256>(mode, a, n_wide, ring, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fmm
