// Clipped sum of a T = 1 layer with at most 16 outputs (a classifier head on its own): gW[o][i] = sum_b c_b zb[b][o] a[b][i].
//
// Bound: latency.  CTA = 64 input columns, lane = two of them, warp w takes rows w, w + 8, ...; the scaled zb of 64 rows wait in
// shared memory, so a row costs a lane one load and 32 multiply-adds.  The fp32-ALU tile kernel ran such a layer on d_in / 64 CTAs
// of serial 16-row steps, with the noise drawn in its epilogue: 256 -> 10, B = 64: 12 to 21 us beside the convolutions of a
// strided CNN, here 4.
#pragma once
#include "kernels_stream.cuh"

namespace dpclip {

constexpr int THIN_OUT = 16, THIN_COLS = 64, THIN_ROWS = 64, THIN_THREADS = 256;
struct ThinParams {
    const void* A; long lda; const void* Z; long ldz;
    int B, d_in, d_out, pairs_ok;          // pairs_ok: two elements of a row of A are one aligned load
    const float* clip;                     // [B] or NULL
    float* gW; long ldg; float* gb;
    float noise_scale; uint32_t k0, k1, sw0, sw1, sb0, sb1;
};

__device__ __forceinline__ float2 thin_load2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 thin_load2(const __nv_bfloat16* p) {
    const uint32_t r = *reinterpret_cast<const uint32_t*>(p);
    return make_float2(__uint_as_float(r << 16), __uint_as_float(r & 0xFFFF0000u));
}

template <typename T>
__global__ void __launch_bounds__(THIN_THREADS)
t1_thin_grad_kernel(const __grid_constant__ ThinParams p) {
    constexpr int WARPS = THIN_THREADS / 32;
    __shared__ __align__(16) float zs[THIN_ROWS][THIN_OUT];
    __shared__ __align__(16) float part[WARPS][THIN_OUT][THIN_COLS];        // 32 KB
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * THIN_COLS + 2 * lane;
    const T* A = static_cast<const T*>(p.A);
    const T* Z = static_cast<const T*>(p.Z);
    float acc[THIN_OUT][2], bias = 0.f;
#pragma unroll
    for (int o = 0; o < THIN_OUT; ++o) acc[o][0] = acc[o][1] = 0.f;
    for (int b0 = 0; b0 < p.B; b0 += THIN_ROWS) {
        // this warp's rows of A are requested before the scaled zb are waited for
        float2 a[THIN_ROWS / WARPS];
#pragma unroll
        for (int k = 0; k < THIN_ROWS / WARPS; ++k) {
            const int b = b0 + warp + k * WARPS;
            a[k] = make_float2(0.f, 0.f);
            if (b < p.B) {
                const T* row = A + (size_t)b * p.lda + c;
                if (p.pairs_ok && c + 1 < p.d_in) a[k] = thin_load2(row);
                else {
                    if (c < p.d_in) a[k].x = to_f32(row[0]);
                    if (c + 1 < p.d_in) a[k].y = to_f32(row[1]);
                }
            }
        }
        if (b0 > 0) __syncthreads();
#pragma unroll
        for (int k = 0; k < THIN_ROWS * THIN_OUT / THIN_THREADS; ++k) {
            const int e = threadIdx.x + k * THIN_THREADS, b = b0 + e / THIN_OUT, o = e % THIN_OUT;
            float z = 0.f;
            if (b < p.B && o < p.d_out) z = (p.clip ? __ldg(p.clip + b) : 1.f) * to_f32(Z[(size_t)b * p.ldz + o]);
            zs[e / THIN_OUT][o] = z;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < THIN_ROWS / WARPS; ++k) {
            if (b0 + warp + k * WARPS >= p.B) break;             // a row that is not there adds nothing, whatever A holds
            const float4* z4 = reinterpret_cast<const float4*>(zs[warp + k * WARPS]);
#pragma unroll
            for (int q = 0; q < THIN_OUT / 4; ++q) {
                const float4 z = z4[q];
                acc[4 * q][0] = fmaf(z.x, a[k].x, acc[4 * q][0]); acc[4 * q][1] = fmaf(z.x, a[k].y, acc[4 * q][1]);
                acc[4 * q + 1][0] = fmaf(z.y, a[k].x, acc[4 * q + 1][0]); acc[4 * q + 1][1] = fmaf(z.y, a[k].y, acc[4 * q + 1][1]);
                acc[4 * q + 2][0] = fmaf(z.z, a[k].x, acc[4 * q + 2][0]); acc[4 * q + 2][1] = fmaf(z.z, a[k].y, acc[4 * q + 2][1]);
                acc[4 * q + 3][0] = fmaf(z.w, a[k].x, acc[4 * q + 3][0]); acc[4 * q + 3][1] = fmaf(z.w, a[k].y, acc[4 * q + 3][1]);
            }
        }
        if (p.gb && blockIdx.x == 0 && threadIdx.x < THIN_OUT) {
#pragma unroll 8
            for (int r = 0; r < THIN_ROWS; ++r) bias += zs[r][threadIdx.x];
        }
    }
#pragma unroll
    for (int o = 0; o < THIN_OUT; ++o) *reinterpret_cast<float2*>(&part[warp][o][2 * lane]) = make_float2(acc[o][0], acc[o][1]);
    if (p.gb && blockIdx.x == 0 && threadIdx.x < THIN_OUT && (int)threadIdx.x < p.d_out) {
        const int o = threadIdx.x;
        if (p.noise_scale > 0.f) {
            float z[4];
            normals_at((size_t)o, p.sb0, p.sb1, p.k0, p.k1, z);
            bias = fmaf(p.noise_scale, z[0], bias);
        }
        p.gb[o] = bias;
    }
    __syncthreads();
    // thread = four columns of one output: the warps' sums in order, the noise, the store
    const int o = threadIdx.x / (THIN_COLS / 4), q = threadIdx.x % (THIN_COLS / 4);
    const int i = blockIdx.x * THIN_COLS + 4 * q;
    if (o >= p.d_out || i >= p.d_in) return;
    float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        const float4 v = *reinterpret_cast<const float4*>(&part[w][o][4 * q]);
        x[0] += v.x; x[1] += v.y; x[2] += v.z; x[3] += v.w;
    }
    if (p.noise_scale > 0.f) {
        float z[4];
        normals_at((size_t)o * p.d_in + i, p.sw0, p.sw1, p.k0, p.k1, z);
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = fmaf(p.noise_scale, z[u], x[u]);
    }
    float* dst = p.gW + (size_t)o * p.ldg + i;
#pragma unroll
    for (int u = 0; u < 4; ++u) if (i + u < p.d_in) dst[u] = x[u];
}

}  // namespace dpclip
