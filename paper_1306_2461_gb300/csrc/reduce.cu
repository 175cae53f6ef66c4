// Reductions over a displacement field for the recirculation-bubble surface of Eq. 3
// (Sect. 3.2): the number of vectors whose streamwise component is at most T_v, and the
// minimum and maximum of a (mean) field, from which T_v = (min + max) / 2.
#include <cooperative_groups.h>
#include <math.h>

#include "of_internal.cuh"

namespace of {

constexpr int RED_THREADS = 256;

// Order-preserving map from float to unsigned (no NaN).
__device__ __forceinline__ unsigned int f2key(float f)
{
    const unsigned int b = __float_as_uint(f);
    return (b >> 31) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key2f(unsigned int k)
{
    return __uint_as_float((k >> 31) ? (k & 0x7fffffffu) : ~k);
}

// What a thread accumulates: the number of values <= Tv ...
struct CountLe {
    float Tv;
    unsigned int c = 0;
    __device__ void take(float v) { c += v <= Tv; }
};
// ... or the smallest and the largest of the values that are numbers: fminf and fmaxf pass a NaN
// over and put -0 before +0, as the order of the keys does. lo > hi when there was no number.
struct MinMax {
    float lo = INFINITY, hi = -INFINITY;
    __device__ void take(float v)
    {
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
};

// Feed p[0..n) to the threads' accumulators: thread t of nt, 16-byte loads where p is aligned
// for them, four in flight per thread.
template <typename A> __device__ __forceinline__ void scan(const float *p, long long n, long long t, long long nt, A &a)
{
    long long i = 0;   // elements taken by 16-byte loads
    if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
        const float4 *q = reinterpret_cast<const float4 *>(p);
        const long long n4 = n / 4;
        long long k = t;
        for (; k + 3 * nt < n4; k += 4 * nt) {
            float4 w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = __ldg(q + k + j * nt);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                a.take(w[j].x);
                a.take(w[j].y);
                a.take(w[j].z);
                a.take(w[j].w);
            }
        }
        for (; k < n4; k += nt) {
            const float4 w = __ldg(q + k);
            a.take(w.x);
            a.take(w.y);
            a.take(w.z);
            a.take(w.w);
        }
        i = 4 * n4;
    }
    for (long long k = i + t; k < n; k += nt) a.take(__ldg(p + k));
}

// The warp's, then the block's accumulator (valid in thread 0).
__device__ __forceinline__ void warp_reduce(CountLe &a) { a.c = __reduce_add_sync(0xffffffffu, a.c); }
__device__ __forceinline__ void warp_reduce(MinMax &a)
{
    a.lo = key2f(__reduce_min_sync(0xffffffffu, f2key(a.lo)));
    a.hi = key2f(__reduce_max_sync(0xffffffffu, f2key(a.hi)));
}
__device__ __forceinline__ uint2 pack(const CountLe &a) { return make_uint2(a.c, 0u); }
__device__ __forceinline__ uint2 pack(const MinMax &a) { return make_uint2(__float_as_uint(a.lo), __float_as_uint(a.hi)); }
__device__ __forceinline__ void unpack(CountLe &a, uint2 v, bool have) { a.c = have ? v.x : 0u; }
__device__ __forceinline__ void unpack(MinMax &a, uint2 v, bool have)
{
    a.lo = have ? __uint_as_float(v.x) : INFINITY;
    a.hi = have ? __uint_as_float(v.y) : -INFINITY;
}
template <typename A> __device__ __forceinline__ void block_reduce(A &a)
{
    __shared__ uint2 s[32];
    const int warps = blockDim.x / 32;
    warp_reduce(a);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = pack(a);
    __syncthreads();
    if (threadIdx.x < 32) {
        unpack(a, s[threadIdx.x], (int)threadIdx.x < warps);
        warp_reduce(a);
    }
}
__device__ __forceinline__ void write_result(const CountLe &a, void *out)
{
    *static_cast<unsigned long long *>(out) = a.c;
}
__device__ __forceinline__ void write_result(const MinMax &a, void *out)
{
    const bool none = a.lo > a.hi;   // the field had no number: NaN
    float *o = static_cast<float *>(out);
    o[0] = none ? __int_as_float(0x7fc00000) : a.lo;
    o[1] = none ? __int_as_float(0x7fc00000) : a.hi;
}

// Fields of at most CLUSTER_MAX values: one launch of one cluster, whose blocks hand their
// results to block 0 through distributed shared memory. Its 8 SMs read about 1 TB/s, so up to a
// few megabytes the launch itself is most of the time and the clearing and decoding launches
// of the other form cost more than the idle SMs (CLUSTER_MAX).
constexpr int CLUSTER = 8, CLUSTER_THREADS = 1024;
template <typename A> __global__ void __launch_bounds__(CLUSTER_THREADS) __cluster_dims__(CLUSTER, 1, 1)
cluster_reduce_kernel(const float *p, long long n, A a, void *out)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ uint2 part[CLUSTER];
    // a block's shared memory may be written from outside once all blocks of the cluster have
    // arrived here, that is, started; the wait is hidden behind the scan
    cluster.barrier_arrive();
    scan(p, n, (long long)blockIdx.x * CLUSTER_THREADS + threadIdx.x, (long long)CLUSTER * CLUSTER_THREADS, a);
    block_reduce(a);
    cluster.barrier_wait();
    if (threadIdx.x == 0) cluster.map_shared_rank(part, 0)[blockIdx.x] = pack(a);
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        unpack(a, part[threadIdx.x % CLUSTER], threadIdx.x < CLUSTER);
        warp_reduce(a);
        if (threadIdx.x == 0) write_result(a, out);
    }
}

// Larger fields: all SMs, the blocks' results combined by atomics on the output.
__global__ void __launch_bounds__(RED_THREADS) count_le_kernel(const float *u, long long n, CountLe a,
                                                                unsigned long long *count)
{
    scan(u, n, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, a);
    block_reduce(a);
    if (threadIdx.x == 0 && a.c) atomicAdd(count, (unsigned long long)a.c);
}

__global__ void minmax_init_kernel(unsigned int *mm)
{
    mm[0] = f2key(INFINITY);
    mm[1] = f2key(-INFINITY);
}

__global__ void __launch_bounds__(RED_THREADS) minmax_kernel(const float *f, long long n, unsigned int *mm)
{
    MinMax a;
    scan(f, n, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, a);
    block_reduce(a);
    if (threadIdx.x == 0) {
        atomicMin(&mm[0], f2key(a.lo));
        atomicMax(&mm[1], f2key(a.hi));
    }
}

__global__ void minmax_decode_kernel(unsigned int *mm)
{
    MinMax a;
    a.lo = key2f(mm[0]);
    a.hi = key2f(mm[1]);
    write_result(a, mm);
}

static int reduce_grid(long long n)
{
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long want = (n + RED_THREADS - 1) / RED_THREADS;
    const long long cap = (long long)sms * 8;
    return (int)(want < cap ? (want < 1 ? 1 : want) : cap);
}

// One cluster up to here. Count and extremes, us per call in a row (one cluster; memset and all
// SMs, init, all SMs and decode): 64^2 4.1, 4.1; 4.2, 9.3; 384 x 1792 6.2, 6.2; 6.0, 9.3; 1024^2 6.2,
// 6.2; 6.2, 9.3; 2048^2 14.4, 12.3; 6.5, 10.3; and one launch for the host to queue instead of two
// and three (both for a 384 x 1792 field from Python: 33.8 -> 26.4 us).
constexpr long long CLUSTER_MAX = 1ll << 20;

}  // namespace of

using namespace of;

extern "C" int of_sbubble_count(const float *u, int32_t H, int32_t W, float Tv, unsigned long long *count,
                                of_stream_t stream)
{
    if (!u || !count || H < 1 || W < 1 || !(Tv == Tv)) return OF_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const long long n = (long long)H * W;
    CountLe a;
    a.Tv = Tv;
    if (n <= CLUSTER_MAX) {
        cluster_reduce_kernel<CountLe><<<CLUSTER, CLUSTER_THREADS, 0, st>>>(u, n, a, count);
    } else {
        if (cudaMemsetAsync(count, 0, sizeof(unsigned long long), st) != cudaSuccess) return OF_ECUDA;
        count_le_kernel<<<reduce_grid(n), RED_THREADS, 0, st>>>(u, n, a, count);
    }
    return cudaGetLastError() == cudaSuccess ? OF_OK : OF_ECUDA;
}

extern "C" int of_field_minmax(const float *field, int32_t H, int32_t W, float *minmax, of_stream_t stream)
{
    if (!field || !minmax || H < 1 || W < 1) return OF_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const long long n = (long long)H * W;
    if (n <= CLUSTER_MAX) {
        cluster_reduce_kernel<MinMax><<<CLUSTER, CLUSTER_THREADS, 0, st>>>(field, n, MinMax(), minmax);
    } else {
        unsigned int *mm = reinterpret_cast<unsigned int *>(minmax);
        minmax_init_kernel<<<1, 1, 0, st>>>(mm);
        minmax_kernel<<<reduce_grid(n), RED_THREADS, 0, st>>>(field, n, mm);
        minmax_decode_kernel<<<1, 1, 0, st>>>(mm);
    }
    return cudaGetLastError() == cudaSuccess ? OF_OK : OF_ECUDA;
}
