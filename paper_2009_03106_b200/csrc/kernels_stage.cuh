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
// The copies of one step are a few to a few dozen MB and mostly stay in the 126 MB L2 until the two stages have read them.
// Columns between the width and ld' need no value: the tensor maps end at the width.
#pragma once
#include "common.cuh"

namespace dpclip {
namespace stage {

enum Kind : int { ROWS = 0, ROWS_TO_F32 = 1, TRANSPOSE = 2, IM2COL = 3 };
constexpr int MAX_JOBS = 32;
constexpr int THREADS = 256;
constexpr int ROWS_UNROLL = 4;                 // 16-byte output chunks per thread
constexpr int TILE = 4096;                     // elements of a transpose tile: 64 x 64, or 128 positions x 32 channels
constexpr int IM_WALK = 16;                    // im2col: positions a thread takes of a long row
constexpr int SMEM_MAX = 160 * 1024;

struct Job {
    int kind, es;                  // es = bytes of an input element
    const void* src; void* dst;
    long src_ld; int dst_ld;       // elements (of the input, of the output)
    int rows, cols;                // output rows and width
    int blk_begin;
    // TRANSPOSE / IM2COL
    int T, tiles_a, tiles_b;       // TRANSPOSE: tiles along T and along M, ct = channels of a tile; IM2COL: channel blocks in tiles_b
    int C, H, W, kh, kw, stride, pad, Wo, ct;
    int n_ex, r_out, vec;          // IM2COL: examples and rows of output positions per CTA (tiles_a of them), ct channels; elements per load
    int part, w_out, tiles_x, lead;      // IM2COL, part: a CTA takes w_out positions of one row (tiles_x of them); columns of the window before the first tap's
    int pitch, plane;              // IM2COL: elements of a row and of a channel of the window
};
// Shared memory of an im2col CTA: places of the columns in the window, the window.
__host__ __device__ inline int im_table(const Job& j) { return (j.ct * j.kh * j.kw + 15) / 16 * 16; }
__host__ __device__ inline int im_tile_elems(const Job& j) { return (j.n_ex * j.ct * j.plane + 7) / 8 * 8; }
// Elements between the channels of a window beyond its rows.  A warp reads one element of each of 32 chunks of columns at a time: the
// channels lie so far apart that these meet as few times as possible on a bank (windows of 16 x 14 pixels in bf16, unpadded: six times;
// 132 examples of 14 x 14 maps, 32 to 256 channels: 91 us of staging, padded 60).
constexpr int IM_MAX_PAD = 15;
inline int im_bank_pad_search(int es, int width, int kh, int kw, int pitch, int plane, int step) {
    const int n = 16 / es, shift = es == 4 ? 0 : 1;
    int chan[256], at[256];                                   // channel of a column, its place in the window
    for (int i = 0, c = 0, ky = 0, kx = 0; i < width; ++i) {
        chan[i] = c; at[i] = c * plane + ky * pitch + kx;
        if (++kx == kw) { kx = 0; if (++ky == kh) { ky = 0; ++c; } }
    }
    int best = 1 << 30, pad = 0;
    for (int b = 0; b <= IM_MAX_PAD && best > n * (es == 4 ? 2 : 1); b += step) {
        int sum = 0;
        for (int e = 0; e < n && sum < best; ++e) {
            uint8_t hits[32] = {0};
            int word[32], most = 0;
            for (int i = e; i < width; i += n) {
                const int w = at[i] >> shift, bank = w & 31;
                if (hits[bank] > 0 && word[bank] == w) continue;
                word[bank] = w;
                if (++hits[bank] > most) most = hits[bank];
            }
            sum += most;
        }
        if (sum < best) { best = sum; pad = b; }
        for (int i = 0; i < width; ++i) at[i] += chan[i] * step;
    }
    return pad;
}
// The search takes 2 us of host time (4000 places on banks), in every step that is not recorded: a thread keeps what it found for the
// last few windows, under all that the search reads.  A step of four convolutions, host time of its plan: 1.6 us without any padding,
// 29.6 with a search for every size tried, 2.0 here.
inline int im_bank_pad(const Job& j) {
    struct Found { int es, width, kh, kw, pitch, plane, step, pad; };
    thread_local Found found[32] = {};
    const int max_width = 32 * (16 / j.es), step = j.part ? j.vec : 1;            // whole loads are stored as one word
    int width = (j.ct < j.C ? j.ct : j.C) * j.kh * j.kw;
    if (width > max_width) width = max_width;
    Found& f = found[((unsigned)j.plane * 0x9E3779B1u + (unsigned)j.pitch * 0x85EBCA6Bu + (unsigned)width * 0xC2B2AE35u) >> 27];
    if (f.es != j.es || f.width != width || f.kh != j.kh || f.kw != j.kw || f.pitch != j.pitch || f.plane != j.plane || f.step != step)
        f = {j.es, width, j.kh, j.kw, j.pitch, j.plane, step, im_bank_pad_search(j.es, width, j.kh, j.kw, j.pitch, j.plane, step)};
    return f.pad;
}
inline size_t im_smem(const Job& j) { return (size_t)im_table(j) * 4 + ((size_t)j.n_ex * j.ct * j.plane + 7) / 8 * 8 * j.es + 16; }
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

// A CTA takes ct channels of r_out rows of output positions (of n_ex whole examples when the maps are small, of w_out positions of one
// row when the rows are long).  The input window
// comes into shared memory once, in loads of up to 16 bytes and with zeros around it, so the gather needs no bounds.  A thread then keeps
// the places of N consecutive columns and walks along a row of positions: a patch element costs one load from shared memory at a
// constant distance from the one before and an Nth of a store, and neighbouring threads write neighbouring 16 bytes.
// Bound: issue slots, then latency.  Window elements taken one by one from the map, with masks, through lines of patch rows in
// shared memory were 16 instructions an element, and so was a window in shared memory with a table look-up an element: 288
// columns of 32768 positions in fp32 16 us either way, here 13 (2.9 TB/s written).  All copies of a CNN of three layers 41 -> 29
// us (fp32, 100 MB), of a strided one in bf16 30 -> 24.
template <typename E, int N, int STRIDE, bool PART>
__device__ __forceinline__ void im2col_rows(const Job& j, const E* tile, const int* off, E* dst, int nb, int nyo, int nxo, int width) {
    const int chunks = (width + N - 1) / N, stride = STRIDE ? STRIDE : j.stride;
    // a thread walks along a whole row of positions, along several of narrow maps, along IM_WALK positions of a part of a row
    const int len = PART ? IM_WALK : j.Wo;
    if (PART) nyo = (nxo + IM_WALK - 1) / IM_WALK;
    const int per = PART || len >= 16 ? 1 : (16 + len - 1) / len, runs = (nyo + per - 1) / per;
    for (int i = threadIdx.x; i < nb * runs * chunks; i += THREADS) {
        const int r = i / chunks, k0 = (i - r * chunks) * N;
        const int e = r / runs, y0 = (r - e * runs) * per, y1 = min(y0 + per, nyo);
        const E* x = tile + e * j.ct * j.plane + y0 * j.stride * (PART ? IM_WALK : j.pitch);
        const E* src[N];
#pragma unroll
        for (int k = 0; k < N; ++k) src[k] = x + off[k0 + k];
        E* out = dst + (size_t)((e * nyo + y0) * len) * j.dst_ld + k0;
        const int n = PART ? min(len, nxo - y0 * len) : len;
        for (int y = y0; y < y1; ++y) {
#pragma unroll 4
            for (int xo = 0; xo < n; ++xo) {
                union { E e[N]; uint4 q; } v;
#pragma unroll
                for (int k = 0; k < N; ++k) v.e[k] = src[k][xo * stride];
                if (N == 1) *out = v.e[0];
                else *reinterpret_cast<uint4*>(out) = v.q;
                out += j.dst_ld;
            }
#pragma unroll
            for (int k = 0; k < N; ++k) src[k] += j.stride * (PART ? IM_WALK : j.pitch);
        }
    }
}

// The window of a map with an odd number of elements: a warp takes a channel, its lanes neighbouring elements, four in flight.  (As
// units of one element, with three divisions each: 16 examples of 24 33 x 31 maps in bf16 14.9 us of staging, here 9.4; 32 of 192 13 x 13
// 18.6, here 13.7.)
template <typename E, bool PART>
__device__ __forceinline__ void im2col_load_elements(const Job& j, const E* src, E* tile, int nb, int nc, int ny, int x_lo) {
    const int row_len = PART ? j.pitch : j.W, x_begin = PART ? x_lo : 0;
    const int lane = threadIdx.x & 31, dy = 32 / row_len, dx = 32 - dy * row_len;
    for (int ec = threadIdx.x >> 5; ec < nb * nc; ec += THREADS / 32) {
        const int e = ec / nc, c = ec - e * nc;
        const E* p = src + (size_t)(e * j.C + c) * j.H * j.W + x_begin;
        E* t = tile + (e * j.ct + c) * j.plane + x_begin - x_lo;
        int y = lane / row_len, x = lane - y * row_len;
        while (y < ny) {
            E a[4];
            int d[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                d[k] = -1;
                if (y < ny && (!PART || (x_begin + x >= 0 && x_begin + x < j.W))) { d[k] = y * j.pitch + x; a[k] = __ldg(p + y * j.W + x); }
                x += dx; y += dy;
                if (x >= row_len) { x -= row_len; ++y; }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) if (d[k] >= 0) t[d[k]] = a[k];
        }
    }
}

template <typename E, bool PART>
__device__ __forceinline__ void im2col_job(const Job& j, int blk, uint8_t* smem) {
    constexpr int VEC = 16 / sizeof(E);
    const int cb = blk % j.tiles_b, row = blk / j.tiles_b, xt = PART ? row % j.tiles_x : 0, at = PART ? row / j.tiles_x : row;
    const int rg = at % j.tiles_a, b0 = at / j.tiles_a * j.n_ex;
    const int Ho = j.T / j.Wo, B = j.rows / j.T, kk = j.kh * j.kw;
    const int nb = min(j.n_ex, B - b0), yo0 = rg * j.r_out, nyo = min(j.r_out, Ho - yo0);
    const int c0 = cb * j.ct, nc = min(j.ct, j.C - c0), width = nc * kk;
    const int PW = j.pitch, plane = j.plane;
    int* off = reinterpret_cast<int*>(smem);                               // [ct * kk, rounded up]
    E* tile = reinterpret_cast<E*>(off + im_table(j));
    const int xo0 = PART ? xt * j.w_out : 0, nxo = PART ? min(j.w_out, j.Wo - xo0) : j.Wo;
    // valid input rows: one contiguous run of a channel
    const int y_lo = yo0 * j.stride - j.pad, y0 = max(y_lo, 0), y1 = min(y_lo + (nyo - 1) * j.stride + j.kh, j.H);
    const int ny = max(y1 - y0, 0);
    // loads of a channel's run: they may cross its rows, the last may go beyond them inside the channel; of a window narrower than
    // the row: row by row, each load inside the row or outside it as a whole (the window begins on a multiple of vec)
    const int x_lo = PART ? xo0 * j.stride - j.pad - j.lead : -j.pad, row_len = PART ? PW : j.W;
    const int vec = j.vec, run = (ny * row_len + vec - 1) / vec, units = vec > 1 ? nb * nc * run : 0;
    const E* src = static_cast<const E*>(j.src) + ((size_t)b0 * j.C + c0) * j.H * j.W + (size_t)y0 * j.W;
    constexpr int UNR = 2;
    union { uint4 q; uint2 d; uint32_t w; E e[VEC]; } v[UNR];
    int to[UNR], x0[UNR], n[UNR];
    auto load = [&](int u0) {
#pragma unroll
        for (int k = 0; k < UNR; ++k) {
            const int u = u0 + k * THREADS;
            to[k] = -1;
            if (u >= units) continue;
            const int ec = u / run, at = (u - ec * run) * vec;
            const int e = ec / nc, c = ec - e * nc, y = at / row_len;
            x0[k] = PART ? x_lo + at - y * row_len : at - y * row_len;
            if (PART && (x0[k] < 0 || x0[k] >= j.W)) continue;
            const E* p = src + (size_t)(e * j.C + c) * j.H * j.W + (PART ? y * j.W + x0[k] : at);
            n[k] = PART ? vec : min(vec, ny * row_len - at);
            to[k] = (e * j.ct + c) * plane + (y0 - y_lo + y) * PW + (PART ? x0[k] - x_lo : j.pad + x0[k]);
            if (vec == VEC) v[k].q = __ldg(reinterpret_cast<const uint4*>(p));
            else if (vec * (int)sizeof(E) == 8) v[k].d = __ldg(reinterpret_cast<const uint2*>(p));
            else v[k].w = __ldg(reinterpret_cast<const uint32_t*>(p));
        }
    };
    load(threadIdx.x);                                                     // on their way while the zeros and the table are written
    {
        uint4* z = reinterpret_cast<uint4*>(tile);
        for (int i = threadIdx.x; i < im_tile_elems(j) / VEC; i += THREADS) z[i] = make_uint4(0, 0, 0, 0);
    }
    for (int i = threadIdx.x; i < im_table(j); i += THREADS) {
        const int c = i / kk, k = i - c * kk, ky = k / j.kw;
        off[i] = i < width ? c * plane + ky * PW + (k - ky * j.kw) + (PART ? j.lead : 0) : 0;   // columns behind the width need no value
    }
    __syncthreads();
    for (int u0 = threadIdx.x; u0 < units; u0 += UNR * THREADS) {
        if (u0 != (int)threadIdx.x) load(u0);
#pragma unroll
        for (int k = 0; k < UNR; ++k) {
            if (to[k] < 0) continue;
            if (PART) {
                if (vec == VEC) *reinterpret_cast<uint4*>(tile + to[k]) = v[k].q;
                else if (vec * (int)sizeof(E) == 8) *reinterpret_cast<uint2*>(tile + to[k]) = v[k].d;
                else *reinterpret_cast<uint32_t*>(tile + to[k]) = v[k].w;
                continue;
            }
            int d = to[k], x = x0[k];
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                if (i >= n[k]) break;
                tile[d] = v[k].e[i];
                ++d;
                if (++x == j.W) { x = 0; d += PW - j.W; }
            }
        }
    }
    if (vec == 1) im2col_load_elements<E, PART>(j, src, tile + (y0 - y_lo) * PW, nb, nc, ny, x_lo);
    __syncthreads();
    // the CTA's patch rows are consecutive
    E* dst = static_cast<E*>(j.dst) + ((size_t)b0 * j.T + yo0 * j.Wo + xo0) * j.dst_ld + c0 * kk;
    if (j.dst_ld % VEC != 0) im2col_rows<E, 1, 0, PART>(j, tile, off, dst, nb, nyo, nxo, width);
    else if (j.stride == 1) im2col_rows<E, VEC, 1, PART>(j, tile, off, dst, nb, nyo, nxo, width);
    else if (j.stride == 2) im2col_rows<E, VEC, 2, PART>(j, tile, off, dst, nb, nyo, nxo, width);
    else im2col_rows<E, VEC, 0, PART>(j, tile, off, dst, nb, nyo, nxo, width);
}
}  // namespace stage

// PARTS: some window is a part of a long row.  A kernel of its own: that code beside the other in one kernel cost spills in both.
template <bool PARTS>
__global__ void __launch_bounds__(stage::THREADS, 6)
stage_operands_kernel(const __grid_constant__ stage::Launch q) {
    using namespace stage;
    extern __shared__ __align__(16) uint8_t stage_smem[];
    for (size_t i = (size_t)blockIdx.x * THREADS + threadIdx.x; i < q.n_clear; i += (size_t)gridDim.x * THREADS) q.clear[i] = 0.f;
    griddep_launch_dependents();
    int k = 0;
    while (k + 1 < q.n && (int)blockIdx.x >= q.job[k + 1].blk_begin) ++k;
    const Job& j = q.job[k];
    const int blk = blockIdx.x - j.blk_begin;
    if (j.kind == ROWS || j.kind == ROWS_TO_F32) rows_job(j, blk);
    else if (j.kind == TRANSPOSE) {
        if (j.es == 2) { if (j.ct == 32) transpose_job<uint16_t, 32>(j, blk, stage_smem); else transpose_job<uint16_t, 64>(j, blk, stage_smem); }
        else { if (j.ct == 32) transpose_job<uint32_t, 32>(j, blk, stage_smem); else transpose_job<uint32_t, 64>(j, blk, stage_smem); }
    }
    else if (PARTS && j.part) { if (j.es == 2) im2col_job<uint16_t, true>(j, blk, stage_smem); else im2col_job<uint32_t, true>(j, blk, stage_smem); }
    else { if (j.es == 2) im2col_job<uint16_t, false>(j, blk, stage_smem); else im2col_job<uint32_t, false>(j, blk, stage_smem); }
}

}  // namespace dpclip
