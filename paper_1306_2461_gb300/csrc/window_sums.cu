// The window-sum step alone (of_window_sums), for every radius: the passes of the iteration tile on
// five given planes. In a file of its own, because the first use of a kernel loads all kernels of
// its file: the first call takes 1.4 ms (226 with
// the kernels of every radius in their files).
#include <mutex>

#include "of_internal.cuh"
#include "of_kernels.cuh"

namespace of {

template <int R>
__global__ void __launch_bounds__(LK_THREADS)
window_sums_kernel(const float *ch, int H, int W, int r, int tiles_x, float *out)
{
    extern __shared__ float4 smem4[];
    float *smem = reinterpret_cast<float *>(smem4);
    const int tile = blockIdx.x;
    const int ty0 = (tile / tiles_x) * LK_TH, tx0 = (tile % tiles_x) * LK_TW;
    const size_t N = (size_t)H * W;
    if constexpr (R == 0) {
        const int RH = LK_TH + 2 * r, RW = LK_TW + 2 * r;
        const int plane = RH * RW;
        float *P = smem, *S = smem + 5 * plane;
        for (int i = threadIdx.x; i < plane; i += blockDim.x) {
            const int ry = i / RW, rx = i - ry * RW;
            const int y = ty0 - r + ry, x = tx0 - r + rx;
            const bool in = y >= 0 && y < H && x >= 0 && x < W;
            for (int c = 0; c < 5; ++c) P[c * plane + i] = in ? ch[c * N + (size_t)y * W + x] : 0.0f;
        }
        __syncthreads();
        box_hsum(P, S, RH, RW, r);
        __syncthreads();
        for (int i = threadIdx.x; i < LK_TH * LK_TW; i += blockDim.x) {
            const int ty = i / LK_TW, tx = i % LK_TW;
            const int y = ty0 + ty, x = tx0 + tx;
            if (y >= H || x >= W) continue;
            float s[5];
            box_vsum(S, RH, r, ty, tx, s);
            for (int c = 0; c < 5; ++c) out[c * N + (size_t)y * W + x] = s[c];
        }
    } else {
        // the planes of the iteration tile: channels (0, 1) and (2, 3) as float2 pairs, 4 alone
        using F = FixedTile<R>;
        float2 *P01 = reinterpret_cast<float2 *>(smem);
        float2 *P23 = P01 + F::PAIR_PLANE;
        float *P4 = reinterpret_cast<float *>(P23 + F::PAIR_PLANE);
        for (int i = threadIdx.x; i < F::RH * F::RWE; i += blockDim.x) {
            const int ry = i / F::RWE, rx = i - ry * F::RWE;
            const int y = ty0 - R + ry, x = tx0 - F::RE + rx;
            const bool in = y >= 0 && y < H && x >= 0 && x < W;
            float c[5];
            for (int k = 0; k < 5; ++k) c[k] = in ? ch[k * N + (size_t)y * W + x] : 0.0f;
            P01[ry * F::RWP2 + rx] = make_float2(c[0], c[1]);
            P23[ry * F::RWP2 + rx] = make_float2(c[2], c[3]);
            P4[ry * F::RWP1 + rx] = c[4];
        }
        __syncthreads();
        box_h_pairs<R, LK_TH>(P01);
        box_h_pairs<R, LK_TH>(P23);
        box_h_single<R, LK_TH>(P4);
        __syncthreads();
        constexpr int VR = v_rows<R, LK_TH>();
        for (int i = threadIdx.x; i < LK_TW * (LK_TH / VR); i += blockDim.x) {
            const int tx = i % LK_TW, g = i / LK_TW;
            const int x = tx0 + tx;
            if (x >= W) continue;
            float2 s01[VR], s23[VR];
            float s4[VR];
            box_v_planes<R, LK_TH>(P01, P23, P4, g, tx, s01, s23, s4);
            for (int j = 0; j < VR; ++j) {
                const int y = ty0 + VR * g + j;
                if (y >= H) break;
                const float s[5] = {s01[j].x, s01[j].y, s23[j].x, s23[j].y, s4[j]};
                for (int c = 0; c < 5; ++c) out[c * N + (size_t)y * W + x] = s[c];
            }
        }
    }
}

template <int R> static cudaError_t ws_launch(const float *ch, int H, int W, int r, float *out, cudaStream_t s)
{
    const int tiles_x = (W + LK_TW - 1) / LK_TW, tiles_y = (H + LK_TH - 1) / LK_TH;
    window_sums_kernel<R><<<tiles_x * tiles_y, LK_THREADS, sizeof(float) * lk_tile_smem_floats<R>(r, false), s>>>(
        ch, H, W, r, tiles_x, out);
    return cudaGetLastError();
}

// Raise the kernels' dynamic shared memory limits on the current device, once.
#define OF_SET_WS(R)                                                                                                    \
    if ((e = cudaFuncSetAttribute((const void *)window_sums_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,    \
                                  (int)sizeof(float) * lk_tile_smem_floats<R>(R == 0 ? MAX_RADIUS : R, false))) !=     \
        cudaSuccess)                                                                                                   \
        return e;
static cudaError_t configure()
{
    static std::mutex mu;
    static bool configured[256];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (configured[dev]) return cudaSuccess;
    OF_SET_WS(0)
    OF_RADII(OF_SET_WS)
    OF_RADII_MORE(OF_SET_WS)
    configured[dev] = true;
    return cudaSuccess;
}

#define OF_CASE_WS(R) \
    case R: return ws_launch<R>(ch, H, W, r, out, s);
cudaError_t launch_window_sums(const float *ch, int H, int W, int r, float *out, cudaStream_t s)
{
    const cudaError_t e = configure();
    if (e != cudaSuccess) return e;
    switch (r) {
        OF_RADII(OF_CASE_WS)
        OF_RADII_MORE(OF_CASE_WS)
    default: return ws_launch<0>(ch, H, W, r, out, s);
    }
}

}  // namespace of
