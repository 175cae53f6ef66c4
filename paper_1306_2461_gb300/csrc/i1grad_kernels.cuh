// The variant of the iteration linearised with the FIRST image's gradient (the FOLKI
// lineage the method of Sect. 2.4 comes from): g1 = central difference of I1 at integer
// pixels, indices clamped, halved. The window matrix [Sa Sb; Sb Sc] = sum over the
// window of g1 g1^T then depends on I1 only: i1_hess_kernel sums it once per level, and
// each iteration forms and sums only the two right-hand-side channels
//     g1 e~,  e~ = I1 - I2(x + u_k) + g1 . (u_k - u_ref),
// then solves [Sa Sb; Sb Sc] (u_{k+1} - u_ref) = sum g1 e~ with the guard of solve2.
#pragma once

#include "of_internal.cuh"
#include "of_kernels.cuh"

namespace of {

// I1 at (x, y) and its central-difference gradient (neighbour indices clamped).
template <bool NC, typename T>
__device__ __forceinline__ void i1_grad(const T *I1, int pitch, int H, int W, int x, int y, float &c, float &gx,
                                        float &gy)
{
    const T *row = I1 + y * pitch;
    c = ldf<NC>(row + x);
    const float xm = ldf<NC>(row + max(x - 1, 0)), xp = ldf<NC>(row + min(x + 1, W - 1));
    const float ym = ldf<NC>(I1 + max(y - 1, 0) * pitch + x), yp = ldf<NC>(I1 + min(y + 1, H - 1) * pitch + x);
    gx = (xp - xm) * 0.5f;
    gy = (yp - ym) * 0.5f;
}

template <int R> inline __host__ __device__ int i1_smem_floats(int r, int channels)
{
    if constexpr (R == 0) {
        const int RH = I1_TH + 2 * r, RW = LK_TW + 2 * r;
        return channels * (RH * RW + RH * LK_TW);
    } else {   // the window matrices: P01 and P4
        using F = FixedTile<R, I1_TH>;
        return 2 * F::PAIR_PLANE + F::RH * F::RWP1;
    }
}

// Window matrix of one level: (Sa, Sb, Sc, 0) at every pixel of one output tile, for any window
// radius r given at run time.
template <typename T>
__device__ __forceinline__ void i1_hess_tile_generic(const HessArgs &a, int tile, int r, float *smem)
{
    const int tyi = tile / a.tiles_x;
    const int ty0 = tyi * I1_TH, tx0 = (tile - tyi * a.tiles_x) * LK_TW;
    const T *I1 = static_cast<const T *>(a.I1);
    const int RH = I1_TH + 2 * r, RW = LK_TW + 2 * r;
    const int plane = RH * RW;
    for (int i = threadIdx.x; i < plane; i += LK_THREADS) {
        const int ry = i / RW, rx = i - ry * RW;
        const int y = ty0 - r + ry, x = tx0 - r + rx;
        float p0 = 0.0f, p1 = 0.0f, p2 = 0.0f;
        if ((unsigned)y < (unsigned)a.H && (unsigned)x < (unsigned)a.W) {
            float c, gx, gy;
            i1_grad<false>(I1, a.pitch, a.H, a.W, x, y, c, gx, gy);
            p0 = gx * gx;
            p1 = gx * gy;
            p2 = gy * gy;
        }
        smem[i] = p0;
        smem[plane + i] = p1;
        smem[2 * plane + i] = p2;
    }
    __syncthreads();
    float *S = smem + 3 * plane;
    box_hsum<3>(smem, S, RH, RW, r);
    __syncthreads();
    for (int i = threadIdx.x; i < I1_TH * LK_TW; i += LK_THREADS) {
        const int ty = i / LK_TW, tx = i - ty * LK_TW;
        const int y = ty0 + ty, x = tx0 + tx;
        if (y >= a.H || x >= a.W) continue;
        float s[3];
        box_vsum<3>(S, RH, r, ty, tx, s);
        a.hess[(size_t)y * a.hess_pitch + x] = make_float4(s[0], s[1], s[2], 0.0f);
    }
}

// The same for a fixed radius: pixel pairs, the first two channels in a pair plane (P01) and the
// third in P4, summed by the passes of the iteration tile. 16 images of 1024^2 at r = 4 take 99 us (302
// MB, 45 us at the memory's rate); one pixel at a time with three planes of floats, 105.
template <typename T, int R>
__device__ __forceinline__ void i1_hess_tile(const HessArgs &a, int tile, float *smem)
{
    using F = FixedTile<R, I1_TH>;
    const int tyi = tile / a.tiles_x;
    const int ty0 = tyi * I1_TH, tx0 = (tile - tyi * a.tiles_x) * LK_TW;
    float2 *P01 = reinterpret_cast<float2 *>(smem);
    float *P4 = smem + 2 * F::PAIR_PLANE;
    const T *I1 = static_cast<const T *>(a.I1);
    constexpr int NPR = F::RWE / 2, RPI = LK_THREADS / NPR;
    const int cx = threadIdx.x % NPR, rs = threadIdx.x / NPR;
    const int x = tx0 - F::RE + 2 * cx;
    const bool inx = (unsigned)x < (unsigned)a.W, inq = (unsigned)(x + 1) < (unsigned)a.W;
    if (rs < RPI) {
#pragma unroll 2
        for (int ry = rs; ry < F::RH; ry += RPI) {
            const int y = ty0 - R + ry;
            float4 s01 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            float2 s4 = f2(0.0f, 0.0f);
            if (inx && (unsigned)y < (unsigned)a.H) {
                float2 c, GX, GY;
                i1_grad_pair<T, false, false>(I1 + (y * a.pitch + x), a.pitch, a.H, a.W, x, y, inq, c, GX, GY);
                const float2 q0 = mul2(GX, GX), q1 = mul2(GX, GY), q2 = mul2(GY, GY);
                s01 = inq ? make_float4(q0.x, q1.x, q0.y, q1.y) : make_float4(q0.x, q1.x, 0.0f, 0.0f);
                s4 = f2(q2.x, inq ? q2.y : 0.0f);
            }
            reinterpret_cast<float4 *>(P01)[ry * (F::RWP2 / 2) + cx] = s01;
            reinterpret_cast<float2 *>(P4)[ry * (F::RWP1 / 2) + cx] = s4;
        }
    }
    __syncthreads();
    box_h_pairs<R, I1_TH>(P01);
    box_h_single<R, I1_TH>(P4);
    __syncthreads();
    constexpr int VR = v_rows<R, I1_TH>(), NV = 2 * R + VR;
    for (int i = threadIdx.x; i < LK_TW * (I1_TH / VR); i += LK_THREADS) {
        const int tx = i % LK_TW, g = i / LK_TW;
        const int xo = tx0 + tx, yb = ty0 + VR * g;
        if (xo >= a.W || yb >= a.H) continue;
        float2 s01[VR];
        float s4[VR];
        {
            float2 v[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) v[q] = P01[(VR * g + q) * F::RWP2 + tx];
            box4v<R, 0>(v, s01);
        }
        {
            float v[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) v[q] = P4[(VR * g + q) * F::RWP1 + tx];
            box4v<R, 0>(v, s4);
        }
#pragma unroll
        for (int j = 0; j < VR; ++j)
            if (yb + j < a.H)
                a.hess[(size_t)(yb + j) * a.hess_pitch + xo] = make_float4(s01[j].x, s01[j].y, s4[j], 0.0f);
    }
}
static_assert(I1_TH % 6 != 0, "four-row groups in the window-matrix tile");

// One iteration of the variant on one output tile, for any window radius r given at run time
// (the fixed radii run the tiles of the main method with the variant's stage 1 and solve).
template <typename T>
__device__ __forceinline__ void i1_iter_tile(const IterArgs &a, int tile, int r, float fp64_cond, float *smem)
{
    const int tyi = tile / a.tiles_x;
    const int ty0 = tyi * I1_TH, tx0 = (tile - tyi * a.tiles_x) * LK_TW;
    const T *I1 = static_cast<const T *>(a.I1);
    const T *I2 = static_cast<const T *>(a.I2);
    const float2 ref = flow_at<false>(a, min(tx0 + LK_TW / 2, a.W - 1), min(ty0 + I1_TH / 2, a.H - 1));
    const int RH = I1_TH + 2 * r, RW = LK_TW + 2 * r;
    const int plane = RH * RW;
    for (int i = threadIdx.x; i < plane; i += LK_THREADS) {
        const int ry = i / RW, rx = i - ry * RW;
        const int y = ty0 - r + ry, x = tx0 - r + rx;
        float p0 = 0.0f, p1 = 0.0f;
        if ((unsigned)y < (unsigned)a.H && (unsigned)x < (unsigned)a.W) {
            const float2 f = flow_at<false>(a, x, y);
            float c, gx, gy;
            i1_grad<false>(I1, a.pitch, a.H, a.W, x, y, c, gx, gy);
            const float Iw = bil_at<false>(I2, a.pitch, a.H, a.W, x, y, f.x, f.y);
            const float e = resid(c, Iw, gx, gy, f.x - ref.x, f.y - ref.y);
            p0 = gx * e;
            p1 = gy * e;
        }
        smem[i] = p0;
        smem[plane + i] = p1;
    }
    __syncthreads();
    float *S = smem + 2 * plane;
    box_hsum<2>(smem, S, RH, RW, r);
    __syncthreads();
    for (int i = threadIdx.x; i < I1_TH * LK_TW; i += LK_THREADS) {
        const int ty = i / LK_TW, tx = i - ty * LK_TW;
        const int y = ty0 + ty, x = tx0 + tx;
        if (y >= a.H || x >= a.W) continue;
        float s[2];
        box_vsum<2>(S, RH, r, ty, tx, s);
        const float4 h = a.hess[(size_t)y * a.hess_pitch + x];
        const float sj[5] = {h.x, h.y, h.z, s[0], s[1]};
        solve_store<false, -1>(a, x, y, ref, fp64_cond, sj);
    }
}

template <typename T, int R>
__global__ void __launch_bounds__(LK_THREADS) i1_hess_kernel(HessArgs a, int r)
{
    extern __shared__ float4 smem4[];
    chain_begin();
    if constexpr (R == 0) i1_hess_tile_generic<T>(a, blockIdx.x, r, reinterpret_cast<float *>(smem4));
    else i1_hess_tile<T, R>(a, blockIdx.x, reinterpret_cast<float *>(smem4));
}

// Resident blocks per SM. The iteration is bound by latency and then by memory (36 bytes per
// pixel): as the main method's single tiles, with one product plane, a level-0 launch of 16 pairs of
// 1024^2 at r = 4 takes 142 us (its bytes 89 us), with tiles of their own that gathered every tap and
// estimate one pixel at a time 188; r = 10 196 instead of 295; a 1024^2 pair 203 -> 155 us. In strips,
// whose tiles shared a reference flow (see ref_group): 153 and 177.
#ifndef OF_I1_MIN_BLOCKS
#define OF_I1_MIN_BLOCKS 5
#endif
template <int R> constexpr int i1_min_blocks() { return R == 0 ? 4 : (R <= 6 ? OF_I1_MIN_BLOCKS : (R <= 12 ? 4 : 3)); }
// The same for the phase launches, whose single tiles fill the SMs (level-0 launch of 16 pairs of 1024^2,
// us, with 5, 6 and 7 blocks at r <= 6, 4, 5 and 6 above): r = 2 146, 151, 150; r = 3 150, 138; r = 4 153, 142,
// 164; r = 6 171, 164, 190; r = 8 194, 181, 176; r = 10 210, 201, 196; r = 12 229, 234, 233; with 3, 4 and 5:
// r = 13 242, 242, 244; r = 16 307, 307, 314. One pair, whose launches do not fill them, is slower with 6
// (r = 4 154 -> 160 us).
template <int R> constexpr int i1_phase_blocks()
{
    return R >= 3 && R <= 10 ? 6 : i1_min_blocks<R>();
}

template <typename T, int R>
__global__ void __launch_bounds__(LK_THREADS, i1_min_blocks<R>())
i1_iter_kernel(const __grid_constant__ IterArgs a, const __grid_constant__ StageMaps m, int r, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    if constexpr (R == 0) {
        chain_begin();
        i1_iter_tile<T>(a, blockIdx.x, r, fp64_cond, smem);
    } else {
        uint32_t phase = 0;
        lk_tile_init<R, LK_TH, LK_TW, false, true>(smem);
        chain_begin();
        lk_tile_fixed<T, false, R, -1, LK_TH, false, LK_THREADS, true>(a, &m, blockIdx.x, fp64_cond, smem, phase);
    }
}

// Small tiles of one pair.
template <typename T, int R>
__global__ void __launch_bounds__(SM_THREADS, i1_min_blocks<R>())
i1_small_kernel(const __grid_constant__ IterArgs a, const __grid_constant__ StageMaps m, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    if constexpr (R != 0) {
        lk_tile_init<R, SM_TH, SM_TW, false, true>(smem);
        chain_begin();
        lk_tile_small<T, false, R, -1, true>(a, &m, blockIdx.x, fp64_cond, smem);
    }
}

// The same over the tiles of up to PHASE_PAIRS pairs (batched form).
template <typename T, int R>
__global__ void __launch_bounds__(LK_THREADS) phase_hess_kernel(const __grid_constant__ HessPhase P, int r)
{
    extern __shared__ float4 smem4[];
    chain_begin();
    const int p = phase_pair(P.prefix, P.npairs, blockIdx.x);
    if constexpr (R == 0) i1_hess_tile_generic<T>(P.a[p], blockIdx.x - P.prefix[p], r, reinterpret_cast<float *>(smem4));
    else i1_hess_tile<T, R>(P.a[p], blockIdx.x - P.prefix[p], reinterpret_cast<float *>(smem4));
}

template <typename T, int R>
__global__ void __launch_bounds__(LK_THREADS, i1_phase_blocks<R>())
phase_i1_iter_kernel(const __grid_constant__ IterPhase P, int r, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    const int p = phase_pair(P.prefix, P.npairs, blockIdx.x);
    const int unit = blockIdx.x - P.prefix[p];
    if constexpr (R == 0) {
        chain_begin();
        i1_iter_tile<T>(P.a[p], unit, r, fp64_cond, smem);
    } else {
        uint32_t phase = 0;
        lk_tile_init<R, LK_TH, LK_TW, false, true>(smem);
        chain_begin();
        const int t2 = blockIdx.x + P.ahead;
        if (P.ahead > 0 && t2 < P.prefix[P.npairs]) {
            const int q = phase_pair(P.prefix, P.npairs, t2);
            prefetch_tile<T, -1, LK_TH>(P.a[q], t2 - P.prefix[q], R);
        }
        lk_tile_fixed<T, false, R, -1, LK_TH, false, LK_THREADS, true>(P.a[p], &P.m[p], unit, fp64_cond, smem, phase);
    }
}

template <typename T, int R>
__global__ void __launch_bounds__(SM_THREADS, i1_min_blocks<R>())
phase_i1_small_kernel(const __grid_constant__ IterPhase P, float fp64_cond)
{
    extern __shared__ __align__(128) float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    if constexpr (R != 0) {
        const int p = phase_pair(P.prefix, P.npairs, blockIdx.x);
        lk_tile_init<R, SM_TH, SM_TW, false, true>(smem);
        chain_begin();
        lk_tile_small<T, false, R, -1, true>(P.a[p], &P.m[p], blockIdx.x - P.prefix[p], fp64_cond, smem);
    }
}

// Dynamic shared memory of the variant's iteration kernels (bytes).
template <int R> inline size_t i1_iter_smem(int r, bool small, bool stage, int elem_bytes)
{
    if constexpr (R == 0) {
        return sizeof(float) * (size_t)i1_smem_floats<0>(r, 2);
    } else {
        using S = FixedTile<R, SM_TH, SM_TW, true>;
        using F = FixedTile<R, LK_TH, LK_TW, true>;
        int f;
        if (small) f = stage ? S::smem_staged(elem_bytes) : S::SMEM_NOSTAGE;
        else f = stage ? F::smem_staged(elem_bytes) : F::SMEM_NOSTAGE;
        return sizeof(float) * (size_t)f;
    }
}

}  // namespace of
