// Small helper kernels around the fused step: layout conversion, m = v^2 dt^2,
// velocity range, receiver gathers and the graph step counter.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace sgb {

struct PadGeom {
    int Nx, Ny, Nz;
    long long sx, sxy, origin;
};

// Layout conversion.  All of it is bound by HBM: 4 bytes in and out per point
// (2 for 16-bit fields).  A block takes CONV_ITEMS items (quads, or single points
// where a quad would be misaligned) of one plane, so the only index arithmetic
// left is one 32-bit division by the row length per item (64-bit divisions of a
// flat index took most of the time before), and each thread has CONV_UNROLL
// loads in flight before its first store.  384 x 384 x 256: pack 222 -> 51 us,
// unpack 124 -> 49 us (323 and 302 MB: 6.3 and 6.1 TB/s); 383 x 381 x 257, point
// by point: 220 -> 77 and 122 -> 60 us.  The items that one launch counts in a
// plane fit 32 bits: rows j0 .. j0 + rows - 1 of every plane, all of them but in
// planes of more than 2^31 items (for_row_slabs).
constexpr int CONV_THREADS = 256, CONV_UNROLL = 4, CONV_ITEMS = CONV_THREADS * CONV_UNROLL;

// Items of V elements: global loads and stores (fp32 and 16-bit).
template <int V>
struct Vec {
    float v[V];
};
__device__ __forceinline__ Vec<4> ld_vec(const float *p, Vec<4> *)
{
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    return {{q.x, q.y, q.z, q.w}};
}
__device__ __forceinline__ Vec<1> ld_vec(const float *p, Vec<1> *) { return {{__ldg(p)}}; }
template <class T>
__device__ __forceinline__ Vec<4> ld_vec(const T *p, Vec<4> *)
{
    const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p));
    const T *e = reinterpret_cast<const T *>(&q);
    return {{(float)e[0], (float)e[1], (float)e[2], (float)e[3]}};
}
template <class T>
__device__ __forceinline__ Vec<1> ld_vec(const T *p, Vec<1> *)
{
    return {{(float)*p}};
}
__device__ __forceinline__ void st_vec(float *p, const Vec<4> &q)
{
    *reinterpret_cast<float4 *>(p) = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
}
template <class T>
__device__ __forceinline__ void st_vec(T *p, const Vec<4> &q)
{
    const T e[4] = {T(q.v[0]), T(q.v[1]), T(q.v[2]), T(q.v[3])};
    *reinterpret_cast<uint2 *>(p) = *reinterpret_cast<const uint2 *>(e);
}
template <class T>
__device__ __forceinline__ void st_vec(T *p, const Vec<1> &q)
{
    *p = T(q.v[0]);
}

// compact fp32 (Nz, Ny, Nx) -> padded field of type T (rounded to nearest), halo
// and row padding zero; padded coordinates (ii, jj, kk) map to computed
// (ii - 8, jj - 4, kk - 4).  V: 4 where Nx is a multiple of 4 and both arrays
// are 16-byte aligned, else 1.  M: the compact array is the velocity model and
// m = (v dt)^2 is stored; range (if any) receives the model's range: [0] max and
// [1] min as float bit patterns (positive floats order like integers), [2]
// counts warps that saw a non-finite or non-positive value.
template <class T, int V, bool M>
__global__ void __launch_bounds__(CONV_THREADS)
    to_padded_kernel(PadGeom g, const float *__restrict__ src, T *__restrict__ dst, float dt,
                     int *range, int j0, int rows)
{
    const uint32_t row = uint32_t(g.sx) / V, items = row * uint32_t(rows);
    float mx = 0.0f, mn = 3.0e38f;
    int bad = 0;
    for (int kk = blockIdx.y; kk < g.Nz + 8; kk += gridDim.y) {
        const bool in_z = kk >= 4 && kk < g.Nz + 4;
        const float *sp = src + (long long)(kk - 4) * g.Ny * g.Nx;
        T *dp = dst + (long long)kk * g.sxy + j0 * g.sx;
        const uint32_t t0 = blockIdx.x * CONV_ITEMS + threadIdx.x;
        Vec<V> val[CONV_UNROLL];
#pragma unroll
        for (int u = 0; u < CONV_UNROLL; ++u) {
            const uint32_t t = t0 + u * CONV_THREADS;
            const uint32_t jj = t / row;
            const int ii = (t - jj * row) * V;
            const int i = ii - 8, j = j0 + int(jj) - 4;
            const bool in = t < items && in_z && i >= 0 && i < g.Nx && j >= 0 && j < g.Ny;
#pragma unroll
            for (int e = 0; e < V; ++e) val[u].v[e] = 0.0f;
            if (in) {
                val[u] = ld_vec(sp + (long long)j * g.Nx + i, (Vec<V> *)nullptr);
                if constexpr (M) {
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                        const float v = val[u].v[e];
                        if (!isfinite(v) || v <= 0.0f) bad = 1;
                        else mx = fmaxf(mx, v), mn = fminf(mn, v);
                        const float w = __fmul_rn(v, dt);
                        val[u].v[e] = __fmul_rn(w, w);
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < CONV_UNROLL; ++u) {
            const uint32_t t = t0 + u * CONV_THREADS;
            if (t < items) st_vec(dp + (long long)t * V, val[u]);
        }
    }
    if constexpr (M) {
        if (!range) return;
        __shared__ int s_mx, s_mn, s_bad;
        if (threadIdx.x == 0) s_mx = 0, s_mn = 0x7f7fffff, s_bad = 0;
        __syncthreads();
        for (int o = 16; o > 0; o >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            bad |= __shfl_xor_sync(0xffffffffu, bad, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&s_mx, __float_as_int(mx));
            atomicMin(&s_mn, __float_as_int(mn));
            if (bad) atomicAdd(&s_bad, 1);
        }
        __syncthreads();
        if (threadIdx.x == 0) {  // most blocks change nothing: look before the atomic
            volatile int *r = range;
            if (s_mx > r[0]) atomicMax(range, s_mx);
            if (s_mn < r[1]) atomicMin(range + 1, s_mn);
            if (s_bad) atomicAdd(range + 2, s_bad);
        }
    }
}

// padded field of type T -> compact fp32, times the field's scale (null: 1).
// V as above.
template <class T, int V>
__global__ void __launch_bounds__(CONV_THREADS)
    from_padded_kernel(PadGeom g, const T *__restrict__ src, const float *scale,
                       float *__restrict__ dst, int j0, int rows)
{
    const uint32_t row = uint32_t(g.Nx) / V, items = row * uint32_t(rows);
    const float s = scale ? *scale : 1.0f;
    for (int k = blockIdx.y; k < g.Nz; k += gridDim.y) {
        const T *sp = src + g.origin + (long long)k * g.sxy + j0 * g.sx;
        float *dp = dst + ((long long)k * g.Ny + j0) * g.Nx;
        const uint32_t t0 = blockIdx.x * CONV_ITEMS + threadIdx.x;
        Vec<V> val[CONV_UNROLL];
#pragma unroll
        for (int u = 0; u < CONV_UNROLL; ++u) {
            const uint32_t t = t0 + u * CONV_THREADS;
            const uint32_t j = t / row, i = (t - j * row) * V;
            if (t < items) val[u] = ld_vec(sp + (long long)j * g.sx + i, (Vec<V> *)nullptr);
        }
#pragma unroll
        for (int u = 0; u < CONV_UNROLL; ++u) {
            const uint32_t t = t0 + u * CONV_THREADS;
            if (scale)
#pragma unroll
                for (int e = 0; e < V; ++e) val[u].v[e] *= s;
            if (t < items) st_vec(dp + (long long)t * V, val[u]);
        }
    }
}

// row[r] = u[off[r]]; flags non-finite samples.
__global__ void gather_kernel(const float *__restrict__ u, const long long *__restrict__ off,
                              int nrec, float *__restrict__ row, int *err)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < nrec) {
        const float v = u[off[r]];
        row[r] = v;
        if (!isfinite(v)) atomicOr(err, 2);
    }
}

template <class T>
__global__ void gather_t_kernel(const T *__restrict__ u, const long long *__restrict__ off, int nrec,
                                const float *scale, float *__restrict__ row, int *err)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < nrec) {
        const float v = (float)u[off[r]] * (scale ? *scale : 1.0f);
        row[r] = v;
        if (!isfinite(v)) atomicOr(err, 2);
    }
}

__global__ void advance_kernel(int *counter, int by)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) *counter += by;
}

}  // namespace sgb
