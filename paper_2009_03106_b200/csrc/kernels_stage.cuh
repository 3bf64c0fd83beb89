// Operand staging: layer inputs that the tensor-core kernels cannot address (rows that are not 16-byte multiples,
// convolutions given by their feature map, dL/dZ held channel-major) are rewritten ONCE per step, all of a model's in
// one launch, as row-major matrices whose rows start on 16-byte boundaries.  The norm and the clipped-sum stage then
// both read the copies through TMA.
//
//   rows       [rows][ld] -> [rows][ld'], same type (or bf16 -> fp32 for T = 1 models, see the dispatch)
//   transpose  [B][M][T]  -> [B*T][ld'] (M = d_out): dL/dZ of a convolution as back-propagation holds it
//   im2col     [B][C][H][W] -> [B*T][ld'], columns (c, ky, kx), zeros for the padding: the patch matrix of Sec.
//              "Convolutional Layers"
//
// Bound: latency of the loads and stores (strided CNN from feature maps, 31 us: load/store pipe and shared memory 30 %, DRAM
// 11 %).  The copies of one step are a few to a few dozen MB and mostly stay in the 126 MB L2 until the two stages have read
// them.  Columns between the width and ld' need no value: the tensor maps end at the width.
#pragma once
#include "common.cuh"

namespace dpclip {
namespace stage {

enum Kind : int { ROWS = 0, ROWS_TO_F32 = 1, TRANSPOSE = 2, IM2COL = 3 };
constexpr int MAX_JOBS = 32;
constexpr int THREADS = 256;
constexpr int ROWS_UNROLL = 4;                 // 16-byte output chunks per thread
constexpr int TILE = 4096;                     // elements of a transpose tile: 64 x 64, or 128 positions x 32 channels
constexpr int IM_MAX_ROWS = 256;               // im2col: patch rows per CTA, 32 to 256
constexpr int SMEM_MAX = 160 * 1024;

struct Job {
    int kind, es;                  // es = bytes of an input element
    const void* src; void* dst;
    long src_ld; int dst_ld;       // elements (of the input, of the output)
    int rows, cols;                // output rows and width
    int blk_begin;
    // TRANSPOSE / IM2COL
    int T, tiles_a, tiles_b;       // TRANSPOSE: tiles along T and along M, ct = channels of a tile; IM2COL: channel blocks in tiles_b
    int C, H, W, kh, kw, stride, pad, Wo, ct, pitch;     // IM2COL: ct channels per CTA, pitch = shared-memory bytes of a patch row
    int cta_rows;                  // IM2COL: patch rows per CTA
};
struct Launch { Job job[MAX_JOBS]; int n, blocks; float* clear; size_t n_clear; };     // clear: fp32 words set to zero by the way

// eight bf16 elements that start at any 2-byte boundary; reads exactly those sixteen bytes
__device__ __forceinline__ uint4 load_bf16x8(const uint16_t* p) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    uint4 v;
    if ((a & 7) == 0) {
        const uint2 lo = __ldg(reinterpret_cast<const uint2*>(p)), hi = __ldg(reinterpret_cast<const uint2*>(p) + 1);
        v = make_uint4(lo.x, lo.y, hi.x, hi.y);
    } else if ((a & 3) == 0) {
        const uint32_t* w = reinterpret_cast<const uint32_t*>(p);
        v = make_uint4(__ldg(w), __ldg(w + 1), __ldg(w + 2), __ldg(w + 3));
    } else {
        const uint32_t* w = reinterpret_cast<const uint32_t*>(p + 1);
        const uint32_t e0 = __ldg(p), w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2), e7 = __ldg(p + 7);
        v = make_uint4(e0 | (w0 << 16), __funnelshift_l(w0, w1, 16), __funnelshift_l(w1, w2, 16), (w2 >> 16) | (e7 << 16));
    }
    return v;
}

__device__ __forceinline__ void rows_job(const Job& j, int blk) {
    const bool cvt = j.kind == ROWS_TO_F32;
    const int per = (j.es == 4 || cvt) ? 4 : 8;              // elements per 16-byte output chunk
    const uint32_t cpr = (uint32_t)j.dst_ld / per;           // chunks per output row
    const uint32_t total = (uint32_t)j.rows * cpr;
    uint4 out[ROWS_UNROLL];
#pragma unroll
    for (int u = 0; u < ROWS_UNROLL; ++u) {
        const uint32_t c = (uint32_t)(blk * ROWS_UNROLL + u) * THREADS + threadIdx.x;
        out[u] = make_uint4(0, 0, 0, 0);
        if (c >= total) continue;
        const uint32_t row = c / cpr;
        const int col = (int)(c - row * cpr) * per;
        const int n = min(per, j.cols - col);
        uint32_t w[4] = {0, 0, 0, 0};
        if (j.es == 4) {
            const uint32_t* p = static_cast<const uint32_t*>(j.src) + (size_t)row * j.src_ld + col;
#pragma unroll
            for (int e = 0; e < 4; ++e) if (e < n) w[e] = __ldg(p + e);
        } else {
            const uint16_t* p = static_cast<const uint16_t*>(j.src) + (size_t)row * j.src_ld + col;
            if (cvt) {
#pragma unroll
                for (int e = 0; e < 4; ++e) if (e < n) w[e] = (uint32_t)__ldg(p + e) << 16;
            } else if (n == 8) {
                const uint4 v = load_bf16x8(p);
                w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) if (e < n) w[e >> 1] |= (uint32_t)__ldg(p + e) << (16 * (e & 1));
            }
        }
        out[u] = make_uint4(w[0], w[1], w[2], w[3]);
    }
#pragma unroll
    for (int u = 0; u < ROWS_UNROLL; ++u) {
        const uint32_t c = (uint32_t)(blk * ROWS_UNROLL + u) * THREADS + threadIdx.x;
        if (c < total) static_cast<uint4*>(j.dst)[c] = out[u];
    }
}

// A tile of positions x channels through shared memory; its rows are 2 elements (bf16) or 1 (fp32) longer than the
// tile, so that neither the writes along T nor the reads along M fall on one bank.  32-channel tiles for narrow layers.
template <typename E, int TM>
__device__ __forceinline__ void transpose_job(const Job& j, int blk, uint8_t* smem) {
    constexpr int TT = TILE / TM, PITCH = TT + 4 / sizeof(E);
    E* tile = reinterpret_cast<E*>(smem);
    const int M = j.cols;
    const int per_ex = j.tiles_a * j.tiles_b;
    const int b = blk / per_ex, r = blk - b * per_ex;
    const int m0 = (r / j.tiles_a) * TM, t0 = (r % j.tiles_a) * TT;
    const E* src = static_cast<const E*>(j.src) + (size_t)b * M * j.T;
    const int tx = threadIdx.x % TT, ty = threadIdx.x / TT;
    constexpr int STEP = THREADS / TT, N = TM / STEP;
    E v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int m = m0 + ty + STEP * i, t = t0 + tx;
        v[i] = (m < M && t < j.T) ? __ldg(src + (size_t)m * j.T + t) : E(0);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) tile[(ty + STEP * i) * PITCH + tx] = v[i];
    __syncthreads();
    constexpr int PER = 16 / sizeof(E), CH = TM / PER;              // 16-byte chunks of a position's channels
#pragma unroll
    for (int k = threadIdx.x; k < TT * CH; k += THREADS) {
        const int c = k % CH, t = k / CH;
        const int m = m0 + c * PER;
        if (t0 + t >= j.T || m >= M) continue;
        union { E e[PER]; uint4 q; } o;
#pragma unroll
        for (int i = 0; i < PER; ++i) o.e[i] = tile[(c * PER + i) * PITCH + t];
        E* dst = static_cast<E*>(j.dst) + ((size_t)b * j.T + t0 + t) * j.dst_ld + m;
        if ((j.dst_ld % PER) == 0) {
            *reinterpret_cast<uint4*>(dst) = o.q;
        } else {
#pragma unroll
            for (int i = 0; i < PER; ++i) if (m + i < M) dst[i] = o.e[i];
        }
    }
}

// cta_rows patch rows x ct channels.  Where a row's window lies and which of its rows and columns are inside the map is
// worked out once per row; then a warp takes (32 rows, channel) at a time -- lane = row, so that neighbouring lanes read
// neighbouring pixels -- and writes the window to kh*kw consecutive elements of the row's line in shared memory; the lines
// leave in 16-byte chunks.  Rows are added until a CTA holds about 36 KB: CTAs of 32 rows of a 3-channel image were all
// latency.
template <typename E>
__device__ __forceinline__ void im2col_job(const Job& j, int blk, uint8_t* smem) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rb = blk / j.tiles_b, cb = blk - rb * j.tiles_b;
    const int row0 = rb * j.cta_rows, c0 = cb * j.ct;
    const int kk = j.kh * j.kw, map = j.H * j.W;
    const int nc = min(j.ct, j.C - c0);
    int2* info = reinterpret_cast<int2*>(smem);                   // [cta_rows]: offset of the window, row and column masks
    uint8_t* lines = smem + IM_MAX_ROWS * sizeof(int2);
    const int b0 = row0 / j.T;
    for (int r = threadIdx.x; r < j.cta_rows; r += THREADS) {
        const int row = row0 + r;
        int2 v = make_int2(0, 0);
        if (row < j.rows) {
            const int b = row / j.T, t = row - b * j.T;
            const int yo = t / j.Wo, xo = t - yo * j.Wo;
            const int y0 = yo * j.stride - j.pad, x0 = xo * j.stride - j.pad;
            uint32_t ym = 0, xm = 0;
            for (int k = 0; k < j.kh; ++k) ym |= (y0 + k >= 0 && y0 + k < j.H) ? 1u << k : 0u;
            for (int k = 0; k < j.kw; ++k) xm |= (x0 + k >= 0 && x0 + k < j.W) ? 1u << k : 0u;
            v = make_int2((b - b0) * j.C * map + y0 * j.W + x0, (int)(ym | xm << 16));
        }
        info[r] = v;
    }
    __syncthreads();
    const E* src = static_cast<const E*>(j.src) + ((size_t)b0 * j.C + c0) * map;
    // a window element is a load and a store of its own size, a chain the kernel waits for: of two channels of bf16 windows of
    // nine the 18 elements leave as nine words (the line of an even channel starts on a word): step of the strided
    // CNN from feature maps 115.1 -> 113.8 us
    constexpr int CH = sizeof(E) == 2 ? 2 : 1;
    const bool nine = j.kh * j.kw == 9 && j.kw == 3;
    const int groups = nine ? (nc + CH - 1) / CH : nc;
    const int pairs = (j.cta_rows >> 5) * groups;
    for (int p = warp; p < pairs; p += THREADS / 32) {
        const int rg = p / groups, ci = (p - rg * groups) * (nine ? CH : 1);
        const int r = rg * 32 + lane;
        const int2 v = info[r];
        const E* x = src + (ptrdiff_t)ci * map + v.x;
        E* line = reinterpret_cast<E*>(lines + r * j.pitch) + ci * kk;
        const uint32_t ym = (uint32_t)v.y & 0xFFFFu, xm = (uint32_t)v.y >> 16;
        if (nine) {
            E e[9 * CH];
            const bool both = ci + CH <= nc;
#pragma unroll
            for (int k = 0; k < 9 * CH; ++k) {
                const int w = k % 9;
                e[k] = ((k < 9 || both) && (ym >> (w / 3) & xm >> (w % 3) & 1u)) ? __ldg(x + (k / 9) * map + (w / 3) * j.W + w % 3) : E(0);
            }
            if (CH == 2 && both) {
#pragma unroll
                for (int k = 0; k < 9; ++k) reinterpret_cast<uint32_t*>(line)[k] = (uint32_t)e[2 * k % (9 * CH)] | (uint32_t)e[(2 * k + 1) % (9 * CH)] << 16;
            } else {
#pragma unroll
                for (int k = 0; k < 9; ++k) line[k] = e[k];
            }
        } else {
            for (int ky = 0, k = 0; ky < j.kh; ++ky)
                for (int kx = 0; kx < j.kw; ++kx, ++k) line[k] = (ym >> ky & xm >> kx & 1u) ? __ldg(x + ky * j.W + kx) : E(0);
        }
    }
    __syncthreads();
    constexpr int PER = 16 / sizeof(E);
    const int width = nc * kk, rows = min(j.cta_rows, j.rows - row0);
    E* dst = static_cast<E*>(j.dst) + (size_t)row0 * j.dst_ld + c0 * kk;
    auto chunk = [&](int r, int c) {
        const uint32_t* s = reinterpret_cast<const uint32_t*>(lines + r * j.pitch + c * 16);
        *reinterpret_cast<uint4*>(dst + (size_t)r * j.dst_ld + c * PER) = make_uint4(s[0], s[1], s[2], s[3]);
    };
    if ((j.dst_ld % PER) == 0) {
        const int cpr = (width + PER - 1) / PER;                  // the last chunk may run into the row's padding
        if (cpr >= 16) {
            for (int r = warp; r < rows; r += THREADS / 32)
                for (int c = lane; c < cpr; c += 32) chunk(r, c);
        } else {
            for (int k = threadIdx.x; k < rows * cpr; k += THREADS) { const int r = k / cpr; chunk(r, k - r * cpr); }
        }
    } else {
        for (int k = threadIdx.x; k < rows * width; k += THREADS) {
            const int r = k / width, c = k - r * width;
            dst[(size_t)r * j.dst_ld + c] = reinterpret_cast<const E*>(lines + r * j.pitch)[c];
        }
    }
}
}  // namespace stage

__global__ void __launch_bounds__(stage::THREADS, 6)
stage_operands_kernel(const __grid_constant__ stage::Launch q) {
    using namespace stage;
    extern __shared__ __align__(16) uint8_t stage_smem[];
    for (size_t i = (size_t)blockIdx.x * THREADS + threadIdx.x; i < q.n_clear; i += (size_t)gridDim.x * THREADS) q.clear[i] = 0.f;
    int k = 0;
    while (k + 1 < q.n && (int)blockIdx.x >= q.job[k + 1].blk_begin) ++k;
    const Job& j = q.job[k];
    const int blk = blockIdx.x - j.blk_begin;
    if (j.kind == ROWS || j.kind == ROWS_TO_F32) rows_job(j, blk);
    else if (j.kind == TRANSPOSE) {
        if (j.es == 2) { if (j.ct == 32) transpose_job<uint16_t, 32>(j, blk, stage_smem); else transpose_job<uint16_t, 64>(j, blk, stage_smem); }
        else { if (j.ct == 32) transpose_job<uint32_t, 32>(j, blk, stage_smem); else transpose_job<uint32_t, 64>(j, blk, stage_smem); }
    }
    else { if (j.es == 2) im2col_job<uint16_t>(j, blk, stage_smem); else im2col_job<uint32_t>(j, blk, stage_smem); }
}

}  // namespace dpclip
