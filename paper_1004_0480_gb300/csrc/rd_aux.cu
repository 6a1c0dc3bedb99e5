// rd_aux.cu -- field packing and FP64 reductions (sm_103a).
#include <cuda_bf16.h>
#include <math.h>

#include "rd_internal.h"

namespace rdk {

namespace {

constexpr int kReduceBlocks = 608;    // fixed: 4 per SM of a 152-SM part
constexpr int kReduceThreads = 256;

template <class ST> __device__ __forceinline__ float to_f(ST v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}
template <class ST> __device__ __forceinline__ ST from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}

struct Held {
    float v[6];
};

// Fields in and out.  A CTA is threads(x) x rows(y), a thread V consecutive
// cells of a row at a time, so there is no division per cell and (V = 4) the
// dense side moves 16 bytes per thread; both passes are bound by HBM.  V = 4
// needs 16-byte rows on the dense side (nx a multiple of 4, aligned base).
// rd_set_field of a 512^3 FP32 field from device memory: 593 us with a copy
// to the staging field and one cell per thread found by 64-bit divisions, 173
// so (158 at the copy rate); 256^3: 96 -> 38, rows of 255 cells 101 -> 67.
template <class ST, int V>
__device__ __forceinline__ void load_cells(const ST* p, float (&v)[V]) {
    if constexpr (V == 1) {
        v[0] = to_f<ST>(*p);
    } else if constexpr (sizeof(ST) == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        const uint2 t = *reinterpret_cast<const uint2*>(p);
        v[0] = __uint_as_float(t.x << 16);
        v[1] = __uint_as_float(t.x & 0xffff0000u);
        v[2] = __uint_as_float(t.y << 16);
        v[3] = __uint_as_float(t.y & 0xffff0000u);
    }
}
template <class ST, int V>
__device__ __forceinline__ void store_cells(ST* p, const float (&v)[V]) {
    if constexpr (V == 1) {
        *p = from_f<ST>(v[0]);
    } else if constexpr (sizeof(ST) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
        __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]);
        __nv_bfloat162 b = __floats2bfloat162_rn(v[2], v[3]);
        *reinterpret_cast<uint2*>(p) =
            make_uint2(*reinterpret_cast<unsigned*>(&a), *reinterpret_cast<unsigned*>(&b));
    }
}

// dense (z, y, x) float32 -> pitched field; held layers take their value
template <class ST, int V>
__global__ void pack_kernel(const float* __restrict__ dense, ST* __restrict__ field, int nx,
                            int ny, int nz, int pitch, unsigned held, Held hv) {
    const long long row = blockIdx.x * (long long)blockDim.y + threadIdx.y;
    if (row >= (long long)ny * nz) return;
    const float* const src = dense + row * nx;
    ST* const dst = field + row * pitch;
    const int z = held ? (int)(row / ny) : 0;
    const int y = held ? (int)(row - (long long)z * ny) : 0;
    for (int x0 = threadIdx.x * V; x0 < nx; x0 += blockDim.x * V) {
        float v[V];
        load_cells<float, V>(src + x0, v);
        if (held) {
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const int x = x0 + e;
                if ((held & 1u) && x == 0) v[e] = hv.v[0];
                else if ((held & 2u) && x == nx - 1) v[e] = hv.v[1];
                else if ((held & 4u) && y == 0) v[e] = hv.v[2];
                else if ((held & 8u) && y == ny - 1) v[e] = hv.v[3];
                else if ((held & 16u) && z == 0) v[e] = hv.v[4];
                else if ((held & 32u) && z == nz - 1) v[e] = hv.v[5];
            }
        }
        store_cells<ST, V>(dst + x0, v);
    }
}

template <class ST, int V>
__global__ void unpack_kernel(const ST* __restrict__ field, float* __restrict__ dense, int nx,
                              int ny, int nz, int pitch) {
    const long long row = blockIdx.x * (long long)blockDim.y + threadIdx.y;
    if (row >= (long long)ny * nz) return;
    const ST* const src = field + row * pitch;
    float* const dst = dense + row * nx;
    for (int x0 = threadIdx.x * V; x0 < nx; x0 += blockDim.x * V) {
        float v[V];
        load_cells<ST, V>(src + x0, v);
        store_cells<float, V>(dst + x0, v);
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// pass 1: block b accumulates rows b, b+G, ... in FP64
template <class ST>
__global__ void __launch_bounds__(kReduceThreads)
reduce_pass1(const ST* __restrict__ field, int nx, int nrows, int pitch,
             double* __restrict__ partials) {
    double s = 0.0, q = 0.0, bad = 0.0;
    for (int row = blockIdx.x; row < nrows; row += gridDim.x) {
        const ST* r = field + (long long)row * pitch;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) {
            const float f = to_f<ST>(r[x]);
            if (isfinite(f)) {
                const double d = (double)f;
                s += d;
                q = fma(d, d, q);
            } else {
                bad += 1.0;
            }
        }
    }
    __shared__ double sh[3][kReduceThreads / 32];
    s = warp_sum(s);
    q = warp_sum(q);
    bad = warp_sum(bad);
    const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (lane == 0) { sh[0][w] = s; sh[1][w] = q; sh[2][w] = bad; }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
        for (int i = 0; i < kReduceThreads / 32; ++i) t += sh[threadIdx.x][i];
        partials[blockIdx.x * 3 + threadIdx.x] = t;
    }
}

// pass 2: one block folds the partials in a fixed order
__global__ void __launch_bounds__(kReduceThreads)
reduce_pass2(const double* __restrict__ partials, int nblocks, double* __restrict__ out) {
    double acc[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
        for (int k = 0; k < 3; ++k) acc[k] += partials[b * 3 + k];
    __shared__ double sh[3][kReduceThreads / 32];
    const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int k = 0; k < 3; ++k) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) sh[k][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
        for (int i = 0; i < kReduceThreads / 32; ++i) t += sh[threadIdx.x][i];
        out[threadIdx.x] = t;
    }
}

// CTA and grid of a pack or unpack over ``rows`` rows of ``vx`` vectors
struct RowShape {
    dim3 block, grid;
    RowShape(long long rows, int vx) {
        int bx = 8;
        while (bx < vx && bx < 256) bx *= 2;
        block = dim3(bx, 256 / bx);
        grid = dim3((unsigned)((rows + block.y - 1) / block.y));
    }
};

bool vectors_fit(const float* dense, int nx) {
    return nx % 4 == 0 && (reinterpret_cast<uintptr_t>(dense) & 15) == 0;
}

template <class ST>
void pack_with(const float* dense, ST* field, int nx, int ny, int nz, int pitch, unsigned held,
               const Held& hv, cudaStream_t st) {
    const long long rows = (long long)ny * nz;
    if (vectors_fit(dense, nx)) {
        const RowShape g(rows, nx / 4);
        pack_kernel<ST, 4><<<g.grid, g.block, 0, st>>>(dense, field, nx, ny, nz, pitch, held, hv);
    } else {
        const RowShape g(rows, nx);
        pack_kernel<ST, 1><<<g.grid, g.block, 0, st>>>(dense, field, nx, ny, nz, pitch, held, hv);
    }
}

template <class ST>
void unpack_with(const ST* field, float* dense, int nx, int ny, int nz, int pitch,
                 cudaStream_t st) {
    const long long rows = (long long)ny * nz;
    if (vectors_fit(dense, nx)) {
        const RowShape g(rows, nx / 4);
        unpack_kernel<ST, 4><<<g.grid, g.block, 0, st>>>(field, dense, nx, ny, nz, pitch);
    } else {
        const RowShape g(rows, nx);
        unpack_kernel<ST, 1><<<g.grid, g.block, 0, st>>>(field, dense, nx, ny, nz, pitch);
    }
}

}  // namespace

cudaError_t launch_pack(const float* dense, char* field, int storage, int nx, int ny, int nz,
                        int pitch, unsigned held_mask, const float* held_val,
                        cudaStream_t st) {
    Held hv;
    for (int i = 0; i < 6; ++i) hv.v[i] = held_val ? held_val[i] : 0.0f;
    if (storage == RD_STORE_F32)
        pack_with(dense, reinterpret_cast<float*>(field), nx, ny, nz, pitch, held_mask, hv, st);
    else
        pack_with(dense, reinterpret_cast<__nv_bfloat16*>(field), nx, ny, nz, pitch, held_mask, hv,
                  st);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const char* field, float* dense, int storage, int nx, int ny, int nz,
                          int pitch, cudaStream_t st) {
    if (storage == RD_STORE_F32)
        unpack_with(reinterpret_cast<const float*>(field), dense, nx, ny, nz, pitch, st);
    else
        unpack_with(reinterpret_cast<const __nv_bfloat16*>(field), dense, nx, ny, nz, pitch, st);
    return cudaGetLastError();
}

int reduce_blocks() { return kReduceBlocks; }

cudaError_t launch_reduce(const char* field, int storage, int nx, int ny, int nz, int pitch,
                          double* partials, double* out, cudaStream_t st) {
    const int nrows = ny * nz;
    if (storage == RD_STORE_F32)
        reduce_pass1<float><<<kReduceBlocks, kReduceThreads, 0, st>>>(
            reinterpret_cast<const float*>(field), nx, nrows, pitch, partials);
    else
        reduce_pass1<__nv_bfloat16><<<kReduceBlocks, kReduceThreads, 0, st>>>(
            reinterpret_cast<const __nv_bfloat16*>(field), nx, nrows, pitch, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    reduce_pass2<<<1, kReduceThreads, 0, st>>>(partials, kReduceBlocks, out);
    return cudaGetLastError();
}

}  // namespace rdk
