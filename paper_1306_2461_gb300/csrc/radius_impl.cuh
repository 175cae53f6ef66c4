// Kernels and launchers for one window radius. Each radius_<R>.cu (the batched launches) and
// pair_<R>.cu (OF_PAIR: the launches of one pair) defines OF_RADIUS and includes this file; radius 0
// is the generic kernel (radius given at run time). Two files, because the first use of a kernel
// loads all kernels of its file.
#pragma once

#include "batch_device.cuh"
#include "i1grad_kernels.cuh"
#include "of_internal.cuh"
#include "of_kernels.cuh"

#ifndef OF_RADIUS
#error "define OF_RADIUS before including radius_impl.cuh"
#endif

namespace of {

// Strips: the phase kernels whose tile height holds the rows carried from tile to tile.
template <int R, int TH> constexpr bool strip_kernel() { return R != 0 && TH >= 2 * R; }
// Radii with every form of the batched launch (0: the run-time-radius kernel); the others
// have the per-pair and phase launches at the default tile height.
template <int R> constexpr bool all_forms() { return R == 0 || radius_specialised(R); }

template <typename T, int R>
__global__ void __launch_bounds__(pair_threads<R>(), lk_min_blocks<R>())
lk_iter_kernel(const __grid_constant__ IterArgs a, const __grid_constant__ StageMaps m, int r, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    uint32_t phase = 0;
    lk_tile_prepare<R>(smem);
    chain_begin();
    lk_tile<T, false, R, -1, LK_TH, false, pair_threads<R>()>(a, &m, blockIdx.x, r, fp64_cond, smem, phase);   // a.strip is 1
}

// The same on small tiles.
template <typename T, int R>
__global__ void __launch_bounds__(SM_THREADS, SM_MIN_BLOCKS)
lk_small_kernel(const __grid_constant__ IterArgs a, const __grid_constant__ StageMaps m, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    if constexpr (R != 0) {
        lk_tile_init<R, SM_TH, SM_TW>(smem);
        chain_begin();
        lk_tile_small<T, false, R, -1>(a, &m, blockIdx.x, fp64_cond, smem);
    }
}

template <typename T, int R>
__global__ void __launch_bounds__(SM_THREADS, SM_MIN_BLOCKS)
phase_small_kernel(const __grid_constant__ IterPhase P, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    if constexpr (R != 0) {
        const int p = phase_pair(P.prefix, P.npairs, blockIdx.x);
        lk_tile_init<R, SM_TH, SM_TW>(smem);
        chain_begin();
        lk_tile_small<T, false, R, -1>(P.a[p], &P.m[p], blockIdx.x - P.prefix[p], fp64_cond, smem);
    }
}

template <int R> int small_smem_floats(bool stage_i2, int elem_bytes)
{
    if constexpr (R == 0) return 0;
    else if (stage_i2) return FixedTile<R, SM_TH, SM_TW>::smem_staged(elem_bytes);
    else return FixedTile<R, SM_TH, SM_TW>::SMEM_NOSTAGE;
}

// One iteration of up to PHASE_PAIRS pairs on one level: block b runs tile
// b - prefix[p] of pair p. The same tile code as lk_iter_kernel, so the same results.
template <typename T, int R, int MODE, int TH>
__global__ void __launch_bounds__(LK_THREADS, lk_min_blocks<R, TH>())
phase_iter_kernel(const __grid_constant__ IterPhase P, int r, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    const int p = phase_pair(P.prefix, P.npairs, blockIdx.x);
    uint32_t phase = 0;
    lk_tile_prepare<R, TH, strip_kernel<R, TH>()>(smem);
    chain_begin();
    if constexpr (R != 0) {
        const int t2 = blockIdx.x + P.ahead;
        if (P.ahead > 0 && t2 < P.prefix[P.npairs]) {
            const int q = phase_pair(P.prefix, P.npairs, t2);
            prefetch_tile<T, MODE, TH>(P.a[q], t2 - P.prefix[q], R);
        }
    }
    lk_tile<T, false, R, MODE, TH, strip_kernel<R, TH>(), LK_THREADS>(P.a[p], &P.m[p], blockIdx.x - P.prefix[p], r, fp64_cond, smem, phase);
}

// The same where no pair is staged, for the radii (5 and 6) at which four blocks per SM fit then and
// three otherwise: 32 pairs of 1024^2 at r = 5 (6), two
// sequences, 3428 (3498) us; with the staged form's three blocks 3727 (3774).
template <int R> constexpr bool gather_kernel()
{
    if constexpr (R == 0) return false;
    else return lk_slots(R) == 3 && 4 * (4 * StripTile<R, LK_TH, false>::SMEM_NOSTAGE + 1024) <= 228 * 1024;
}
template <typename T, int R>
__global__ void __launch_bounds__(LK_THREADS, 4) phase_gather_kernel(const __grid_constant__ IterPhase P, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    if constexpr (gather_kernel<R>()) {
        const int p = phase_pair(P.prefix, P.npairs, blockIdx.x);
        chain_begin();
        const int t2 = blockIdx.x + P.ahead;
        if (P.ahead > 0 && t2 < P.prefix[P.npairs]) {
            const int q = phase_pair(P.prefix, P.npairs, t2);
            prefetch_tile<T, -1, LK_TH>(P.a[q], t2 - P.prefix[q], R);
        }
        uint32_t phase = 0;
        lk_tile_fixed<T, false, R, -1, LK_TH, true, LK_THREADS, false, false>(
            P.a[p], nullptr, blockIdx.x - P.prefix[p], fp64_cond, reinterpret_cast<float *>(smem4), phase);
    }
}

// Two same-level iterations of up to PHASE_PAIRS pairs in one launch (iteration fusion
// depth 2): block b runs both on tile b - prefix[p] of pair p (tile height LK_TH).
template <int R> constexpr int fused2_min_blocks()
{
    if constexpr (R == 0) {
        return 1;
    } else {
        constexpr int b = 233472 / (4 * Fused2<R, LK_TH>::SMEM_FLOATS + 1024);
        return b < 1 ? 1 : (b > 2 ? 2 : b);
    }
}
template <typename T, int R>
__global__ void __launch_bounds__(LK_THREADS, fused2_min_blocks<R>())
phase_iter2_kernel(const __grid_constant__ IterPhase P, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    if constexpr (R != 0) {
        const int p = phase_pair(P.prefix, P.npairs, blockIdx.x);
        chain_begin();
        lk_tile_fused2<T, false, R, LK_TH>(P.a[p], blockIdx.x - P.prefix[p], fp64_cond,
                                          reinterpret_cast<float *>(smem4));
    }
}

template <int R> size_t radius_smem_bytes(int r, bool stage_i2)
{
    size_t lk = sizeof(float) * (size_t)lk_tile_smem_floats<R>(r, stage_i2);
    const size_t st = sizeof(float) * (size_t)lk_tile_smem_floats<R, LK_TH, strip_kernel<R, LK_TH>()>(r, stage_i2);
    if (st > lk) lk = st;
    size_t pyr = sizeof(float) * (size_t)PYR_SMEM_FLOATS;
    const size_t zn = sizeof(float) * (size_t)ZN_SMEM_FLOATS;
    if (zn > pyr) pyr = zn;
    return lk > pyr ? lk : pyr;
}

template <typename T, int R>
static cudaError_t lk_for(const IterArgs &a, const StageMaps &m, int r, float fp64_cond, bool small, cudaStream_t s)
{
    if constexpr (R != 0) {
        if (small) {
            return launch_chained(lk_small_kernel<T, R>, a.tiles, SM_THREADS, sizeof(float) * small_smem_floats<R>(a.stage_i2 != 0, (int)sizeof(T)), s, a, m, fp64_cond);
        }
    }
    return launch_chained(lk_iter_kernel<T, R>, a.tiles, pair_threads<R>(), sizeof(float) * lk_tile_smem_floats<R>(r, a.stage_i2 != 0, (int)sizeof(T)), s, a, m, r, fp64_cond);
}

template <int R>
cudaError_t lk_launch(const IterArgs &a, const StageMaps &m, int elem, int r, float fp64_cond, bool small,
                      cudaStream_t s)
{
    switch (elem) {
    case ET_U8: return lk_for<uint8_t, R>(a, m, r, fp64_cond, small, s);
    case ET_U16: return lk_for<uint16_t, R>(a, m, r, fp64_cond, small, s);
    case ET_F32: return lk_for<float, R>(a, m, r, fp64_cond, small, s);
    case ET_F16: return lk_for<__half, R>(a, m, r, fp64_cond, small, s);
    default: return lk_for<__nv_bfloat16, R>(a, m, r, fp64_cond, small, s);
    }
}

// The flow mode is the same for every pair of a phase: at the default tile height one kernel per
// mode (for the radii with fewer forms one for both modes of a level's first iteration; with
// that 64 pairs of 1024^2 at r = 4 take 4883 instead of 4840 us). The other tile height and the
// small tiles read the mode at run time. Fewer kernels keep the build short.
template <int R, int TH> constexpr int phase_mode(int mode)
{
    return TH != LK_TH ? -1 : (mode == FLOW_SAME || all_forms<R>() ? mode : (int)FLOW_FIRST);
}
template <typename T, int R, int TH>
static cudaError_t phase_for_th(const IterPhase &P, int r, float fp64_cond, cudaStream_t s)
{
    bool stage = false;   // shared memory for the staged window if any pair stages
    for (int i = 0; i < P.npairs; ++i) stage = stage || P.a[i].stage_i2 != 0;
    const size_t smem = sizeof(float) * lk_tile_smem_floats<R, TH, strip_kernel<R, TH>()>(r, stage, (int)sizeof(T));
    const int blocks = P.prefix[P.npairs];
    if constexpr (TH == LK_TH && gather_kernel<R>())
        if (!stage)
            return launch_chained(phase_gather_kernel<T, R>, blocks, LK_THREADS,
                                  sizeof(float) * StripTile<R, TH, false>::SMEM_NOSTAGE, s, P, fp64_cond);
    switch (P.a[0].mode) {
    case FLOW_ZERO:
        return launch_chained(phase_iter_kernel<T, R, phase_mode<R, TH>(FLOW_ZERO), TH>, blocks, LK_THREADS, smem, s, P, r,
                              fp64_cond);
    case FLOW_SAME:
        return launch_chained(phase_iter_kernel<T, R, phase_mode<R, TH>(FLOW_SAME), TH>, blocks, LK_THREADS, smem, s, P, r,
                              fp64_cond);
    default:
        return launch_chained(phase_iter_kernel<T, R, phase_mode<R, TH>(FLOW_UPSAMPLE), TH>, blocks, LK_THREADS, smem, s, P,
                              r, fp64_cond);
    }
}

template <typename T, int R>
static cudaError_t phase_for(const IterPhase &P, int r, float fp64_cond, int tile_h, cudaStream_t s)
{
    if constexpr (R != 0) {
        if (tile_h == SM_TH) {
            bool stage = false;
            for (int i = 0; i < P.npairs; ++i) stage = stage || P.a[i].stage_i2 != 0;
            const size_t smem = sizeof(float) * small_smem_floats<R>(stage, (int)sizeof(T));
            const int blocks = P.prefix[P.npairs];
            return launch_chained(phase_small_kernel<T, R>, blocks, SM_THREADS, smem, s, P, fp64_cond);
        }
        if constexpr (all_forms<R>())
            if (tile_h == ALT_TH) return phase_for_th<T, R, ALT_TH>(P, r, fp64_cond, s);
    }
    return phase_for_th<T, R, LK_TH>(P, r, fp64_cond, s);
}

template <int R>
cudaError_t phase_launch(const IterPhase &P, int elem, int r, float fp64_cond, int tile_h, cudaStream_t s)
{
    if (P.prefix[P.npairs] == 0) return cudaSuccess;
    switch (elem) {
    case ET_U8: return phase_for<uint8_t, R>(P, r, fp64_cond, tile_h, s);
    case ET_U16: return phase_for<uint16_t, R>(P, r, fp64_cond, tile_h, s);
    case ET_F32: return phase_for<float, R>(P, r, fp64_cond, tile_h, s);
    case ET_F16: return phase_for<__half, R>(P, r, fp64_cond, tile_h, s);
    default: return phase_for<__nv_bfloat16, R>(P, r, fp64_cond, tile_h, s);
    }
}

template <int R> size_t fused2_smem_bytes()
{
    if constexpr (R == 0) return 0;
    else return sizeof(float) * (size_t)Fused2<R, LK_TH>::SMEM_FLOATS;
}

template <typename T, int R> static cudaError_t phase2_for(const IterPhase &P, float fp64_cond, cudaStream_t s)
{
    return launch_chained(phase_iter2_kernel<T, R>, P.prefix[P.npairs], LK_THREADS, fused2_smem_bytes<R>(), s, P, fp64_cond);
}

template <int R> cudaError_t phase2_launch(const IterPhase &P, int elem, float fp64_cond, cudaStream_t s)
{
    if constexpr (R == 0 || !all_forms<R>()) {
        return cudaErrorInvalidValue;   // fusion needs a fixed-radius kernel
    } else {
        if (P.prefix[P.npairs] == 0) return cudaSuccess;
        switch (elem) {
        case ET_U8: return phase2_for<uint8_t, R>(P, fp64_cond, s);
        case ET_U16: return phase2_for<uint16_t, R>(P, fp64_cond, s);
        case ET_F32: return phase2_for<float, R>(P, fp64_cond, s);
        case ET_F16: return phase2_for<__half, R>(P, fp64_cond, s);
        default: return phase2_for<__nv_bfloat16, R>(P, fp64_cond, s);
        }
    }
}

template <typename T, int R> static cudaError_t i1h_for(const HessArgs &a, int r, cudaStream_t s)
{
    return launch_chained(i1_hess_kernel<T, R>, a.tiles, LK_THREADS, sizeof(float) * i1_smem_floats<R>(r, 3), s, a, r);
}

template <int R> cudaError_t i1h_launch(const HessArgs &a, int elem, int r, cudaStream_t s)
{
    switch (elem) {
    case ET_U8: return i1h_for<uint8_t, R>(a, r, s);
    case ET_U16: return i1h_for<uint16_t, R>(a, r, s);
    case ET_F32: return i1h_for<float, R>(a, r, s);
    case ET_F16: return i1h_for<__half, R>(a, r, s);
    default: return i1h_for<__nv_bfloat16, R>(a, r, s);
    }
}

template <typename T, int R>
static cudaError_t i1_for(const IterArgs &a, const StageMaps &m, int r, float fp64_cond, bool small, cudaStream_t s)
{
    const size_t smem = i1_iter_smem<R>(r, small, a.stage_i2 != 0, (int)sizeof(T));
    if constexpr (R != 0)
        if (small) return launch_chained(i1_small_kernel<T, R>, a.tiles, SM_THREADS, smem, s, a, m, fp64_cond);
    return launch_chained(i1_iter_kernel<T, R>, a.tiles, LK_THREADS, smem, s, a, m, r, fp64_cond);
}

template <int R> cudaError_t i1_launch(const IterArgs &a, const StageMaps &m, int elem, int r, float fp64_cond, bool small, cudaStream_t s)
{
    switch (elem) {
    case ET_U8: return i1_for<uint8_t, R>(a, m, r, fp64_cond, small, s);
    case ET_U16: return i1_for<uint16_t, R>(a, m, r, fp64_cond, small, s);
    case ET_F32: return i1_for<float, R>(a, m, r, fp64_cond, small, s);
    case ET_F16: return i1_for<__half, R>(a, m, r, fp64_cond, small, s);
    default: return i1_for<__nv_bfloat16, R>(a, m, r, fp64_cond, small, s);
    }
}

template <typename T, int R> static cudaError_t phase_hess_for(const HessPhase &P, int r, cudaStream_t s)
{
    return launch_chained(phase_hess_kernel<T, R>, P.prefix[P.npairs], LK_THREADS, sizeof(float) * i1_smem_floats<R>(r, 3), s, P, r);
}

template <int R> cudaError_t phase_hess_launch(const HessPhase &P, int elem, int r, cudaStream_t s)
{
    if (P.prefix[P.npairs] == 0) return cudaSuccess;
    switch (elem) {
    case ET_U8: return phase_hess_for<uint8_t, R>(P, r, s);
    case ET_U16: return phase_hess_for<uint16_t, R>(P, r, s);
    case ET_F32: return phase_hess_for<float, R>(P, r, s);
    case ET_F16: return phase_hess_for<__half, R>(P, r, s);
    default: return phase_hess_for<__nv_bfloat16, R>(P, r, s);
    }
}

template <typename T, int R>
static cudaError_t phase_i1_for(const IterPhase &P, int r, float fp64_cond, int tile_h, cudaStream_t s)
{
    bool stage = false;
    for (int i = 0; i < P.npairs; ++i) stage = stage || P.a[i].stage_i2 != 0;
    const bool small = R != 0 && tile_h == SM_TH;
    const size_t smem = i1_iter_smem<R>(r, small, stage, (int)sizeof(T));
    const int blocks = P.prefix[P.npairs];
    if constexpr (R != 0)
        if (small) return launch_chained(phase_i1_small_kernel<T, R>, blocks, SM_THREADS, smem, s, P, fp64_cond);
    return launch_chained(phase_i1_iter_kernel<T, R>, blocks, LK_THREADS, smem, s, P, r, fp64_cond);
}

template <int R> cudaError_t phase_i1_launch(const IterPhase &P, int elem, int r, float fp64_cond, int tile_h, cudaStream_t s)
{
    if (P.prefix[P.npairs] == 0) return cudaSuccess;
    switch (elem) {
    case ET_U8: return phase_i1_for<uint8_t, R>(P, r, fp64_cond, tile_h, s);
    case ET_U16: return phase_i1_for<uint16_t, R>(P, r, fp64_cond, tile_h, s);
    case ET_F32: return phase_i1_for<float, R>(P, r, fp64_cond, tile_h, s);
    case ET_F16: return phase_i1_for<__half, R>(P, r, fp64_cond, tile_h, s);
    default: return phase_i1_for<__nv_bfloat16, R>(P, r, fp64_cond, tile_h, s);
    }
}

// The tensor maps of the staged fixed-radius tile of height TH: the estimate in boxes
// of the tile's region (RWP2 x RH elements of 8 bytes) and I2 in boxes of the window.
template <int R, int TH, int TW = LK_TW> static bool stage_maps_th(const IterArgs &a, StageMaps &m, int elem, bool strips)
{
    using F = FixedTile<R, TH, TW>;
    const int S = elem_bytes(elem);
    // a window that leaves one block per SM where two would fit gathered (r = 16, and r = 13
    // on with 4-byte levels) costs more than it saves: eight 1024^2 pairs at r = 16 3147 us
    // staged, 2574 gathered
    constexpr int SM_BYTES = 228 * 1024, BLOCK_BYTES = 1024;   // shared memory per SM, and reserved per block
    if (!a.hess && 2 * (4 * F::smem_staged(S) + BLOCK_BYTES) > SM_BYTES && 2 * (4 * F::SMEM_NOSTAGE + BLOCK_BYTES) <= SM_BYTES)
        return false;
    int flow_rows = F::FLOW_BH;
    if constexpr (TW == LK_TW && strip_kernel<R, TH>())
        if (strips) flow_rows = StripTile<R, TH>::BOX;
    if (a.mode == FLOW_SAME &&
        !encode_tile_map(&m.flow, ET_FLOW2, a.fin, a.W, a.H, (size_t)a.fin_pitch * 8, F::RWP2, flow_rows))
        return false;
    return encode_tile_map(&m.i2, elem, a.I2, a.W, a.H, (size_t)a.pitch * S, F::win_w(S), F::WIN_H);
}

template <int R> bool radius_stage_maps(const IterArgs &a, StageMaps &m, int elem, int tile_h, bool strips)
{
    if constexpr (R == 0) {
        return false;
    } else {
        if (tile_h == SM_TH) return stage_maps_th<R, SM_TH, SM_TW>(a, m, elem, strips);
        return tile_h == ALT_TH && all_forms<R>() ? stage_maps_th<R, ALT_TH>(a, m, elem, strips) : stage_maps_th<R, LK_TH>(a, m, elem, strips);
    }
}

template <int R> void *batch_kernel_ptr(int in_format, int storage)
{
    if (in_format == OF_U8) {
        if (storage == OF_F32) return (void *)batch_kernel<uint8_t, float, R>;
        if (storage == OF_F16) return (void *)batch_kernel<uint8_t, __half, R>;
        return (void *)batch_kernel<uint8_t, __nv_bfloat16, R>;
    }
    if (storage == OF_F32) return (void *)batch_kernel<uint16_t, float, R>;
    if (storage == OF_F16) return (void *)batch_kernel<uint16_t, __half, R>;
    return (void *)batch_kernel<uint16_t, __nv_bfloat16, R>;
}

// Raise the dynamic shared memory limit of this radius's kernels of one pair (pair_configure) and of
// the batched launches (batch_configure) on the current device.
#define OF_SET(fn, n) \
    if ((e = cudaFuncSetAttribute((const void *)(fn), cudaFuncAttributeMaxDynamicSharedMemorySize, n)) != cudaSuccess) return e;
#define OF_SET_ALL(K, n) \
    OF_SET((K<uint8_t, R>), n) OF_SET((K<uint16_t, R>), n) OF_SET((K<float, R>), n) OF_SET((K<__half, R>), n) OF_SET((K<__nv_bfloat16, R>), n)
template <int R> cudaError_t pair_configure()
{
    const int r = R == 0 ? MAX_RADIUS : R;
    const int bytes = (int)radius_smem_bytes<R>(r, true), ib = (int)i1_iter_smem<R>(r, false, true, 4);
    const int hb = (int)sizeof(float) * i1_smem_floats<R>(r, 3);
    cudaError_t e;
    OF_SET_ALL(lk_iter_kernel, bytes)
    OF_SET_ALL(i1_hess_kernel, hb)
    OF_SET_ALL(i1_iter_kernel, ib)
    if constexpr (R != 0) {   // small tiles
        const int sb = (int)sizeof(float) * small_smem_floats<R>(true, 4);
        OF_SET_ALL(lk_small_kernel, sb)
        OF_SET_ALL(i1_small_kernel, ib)
    }
    return cudaSuccess;
}

template <int R> cudaError_t batch_configure()
{
    const int r = R == 0 ? MAX_RADIUS : R;
    const int bytes = (int)radius_smem_bytes<R>(r, true), ib = (int)i1_iter_smem<R>(r, false, true, 4);
    const int hb = (int)sizeof(float) * i1_smem_floats<R>(r, 3);
    cudaError_t e;
#define OF_SET_PH(T) \
    OF_SET((phase_iter_kernel<T, R, phase_mode<R, LK_TH>(FLOW_ZERO), LK_TH>), bytes) \
    OF_SET((phase_iter_kernel<T, R, FLOW_SAME, LK_TH>), bytes) \
    OF_SET((phase_iter_kernel<T, R, phase_mode<R, LK_TH>(FLOW_UPSAMPLE), LK_TH>), bytes)
    OF_SET_PH(uint8_t)
    OF_SET_PH(uint16_t)
    OF_SET_PH(float)
    OF_SET_PH(__half)
    OF_SET_PH(__nv_bfloat16)
#undef OF_SET_PH
    OF_SET_ALL(phase_hess_kernel, hb)
    OF_SET_ALL(phase_i1_iter_kernel, ib)
    if constexpr (R != 0) {
        const int sb = (int)sizeof(float) * small_smem_floats<R>(true, 4);
        OF_SET_ALL(phase_small_kernel, sb)
        OF_SET_ALL(phase_i1_small_kernel, ib)
    }
    if constexpr (gather_kernel<R>()) {
        const int gb = (int)sizeof(float) * StripTile<R, LK_TH, false>::SMEM_NOSTAGE;
        OF_SET_ALL(phase_gather_kernel, gb)
    }
    if constexpr (R != 0 && all_forms<R>()) {   // the other tile height, the fused iterations
        const int alt = (int)sizeof(float) * lk_tile_smem_floats<R, ALT_TH, strip_kernel<R, ALT_TH>()>(R, true);
        const int fb = (int)fused2_smem_bytes<R>();
        OF_SET((phase_iter_kernel<uint8_t, R, -1, ALT_TH>), alt)
        OF_SET((phase_iter_kernel<uint16_t, R, -1, ALT_TH>), alt)
        OF_SET((phase_iter_kernel<float, R, -1, ALT_TH>), alt)
        OF_SET((phase_iter_kernel<__half, R, -1, ALT_TH>), alt)
        OF_SET((phase_iter_kernel<__nv_bfloat16, R, -1, ALT_TH>), alt)
        OF_SET_ALL(phase_iter2_kernel, fb)
    }
    if constexpr (all_forms<R>())
        for (int f = 0; f < 2; ++f)
            for (int st = 0; st < 3; ++st) {
                OF_SET(batch_kernel_ptr<R>(f, st), bytes)
            }
    return cudaSuccess;
}
#undef OF_SET_ALL
#undef OF_SET

#ifdef OF_PAIR
template cudaError_t lk_launch<OF_RADIUS>(const IterArgs &, const StageMaps &, int, int, float, bool, cudaStream_t);
template cudaError_t i1h_launch<OF_RADIUS>(const HessArgs &, int, int, cudaStream_t);
template cudaError_t i1_launch<OF_RADIUS>(const IterArgs &, const StageMaps &, int, int, float, bool, cudaStream_t);
template bool radius_stage_maps<OF_RADIUS>(const IterArgs &, StageMaps &, int, int, bool);
template cudaError_t pair_configure<OF_RADIUS>();
#else
template cudaError_t phase_launch<OF_RADIUS>(const IterPhase &, int, int, float, int, cudaStream_t);
template cudaError_t phase_hess_launch<OF_RADIUS>(const HessPhase &, int, int, cudaStream_t);
template cudaError_t phase_i1_launch<OF_RADIUS>(const IterPhase &, int, int, float, int, cudaStream_t);
template cudaError_t phase2_launch<OF_RADIUS>(const IterPhase &, int, float, cudaStream_t);
#ifndef OF_RADIUS_MORE   // one of OF_RADII_MORE
template void *batch_kernel_ptr<OF_RADIUS>(int, int);
#endif
template size_t radius_smem_bytes<OF_RADIUS>(int, bool);
template cudaError_t batch_configure<OF_RADIUS>();
#endif

}  // namespace of
