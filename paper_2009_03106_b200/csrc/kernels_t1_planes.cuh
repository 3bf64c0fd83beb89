// The step of a model of T = 1 layers in two launches (few tiles, or no room in the workspace: the one cooperative launch of
// kernels_fused_t1_tf32.cuh).
//
//   t1_prepare_kernel : CTA = example.  Closed-form norms of all its layers (Sec. "Fully-connected Layers"), its factor, and then its
//                       rows as the tensor cores take them: c zb rounded to bf16 (bf16 models), or c zb and a as three bf16
//                       terms each, x = b0 + b1 + b2 exactly (fp32 models), in the workspace.
//   t1_planes_kernel  : gW = (c Zb)^T A for every layer, 128 x 128 output tiles, K = B rows, noise added, stored once.  Nothing is left
//                       to prepare on the way: TMA -> MMA -> epilogue.
//
// Why.  Inside one launch every tile of A met its Zb tile raw, so diag(c), the low planes and a barrier round trip were paid once per
// tile and stage, d_in / 128 times over (4096 -> 4096 -> 1000, B = 256, bf16: 0.4 us a stage of 32 rows where the MMAs need 0.07);
// and every CTA waited at a grid-wide barrier for the norms, which an example's own CTA knows by itself.
//
// Numbers.  bf16: the same single rounding of c zb as before.  fp32: six products b0 b0, b0 b1, b1 b0, b1 b1, b0 b2, b2 b0 of
// 16-bit operands in place of three tf32 products: as long on the tensor core by the book, but the MN-major layout feeds 16-bit
// operands at full rate (see kernels_group.cuh); windows of 48 additions as before.
//
// Bound: wide models by the L2 -> SM stream of the tiles and the stores of gW (84 MB of outputs, 1280 tiles of 128 KB in bf16: 25 us
// of the second launch) and, with noise, by its generator (45 us, 21 million normals); models of one tile per SM by the chain of the two
// launches (784-1000-1000-10, B = 128, fp32: 5 us and 8).
#pragma once
#include "kernels_fused_t1_tf32.cuh"
#include "kernels_group.cuh"

namespace dpclip {
namespace tc {
namespace t1p {
using f1::BM;
using f1::BN;
using f1::decode;
using f1::Item;
constexpr int NBUF = 2;
// Warps of an example's CTA: sixteen while the CTAs are few, eight beyond (more examples on an SM, fewer idle warps at the barriers).  Step, sixteen
// / eight: 1024-1024-1024 in bf16, B = 256: 11.1 / 10.9 us, 512: 15.2 / 12.5, 2048: 38 / 28; 784-1000-1000-10 in fp32, 256: 16.3 / 16.6, 512:
// 25.5 / 22.8, 2048: 82.6 / 75.4 (one cooperative launch 78.2).
constexpr int PREP_FEW_EXAMPLES = 296, CHUNK = 512;               // CHUNK: elements a warp takes at a time
constexpr int N_EPILOGUE_WARPS = 16, N_BIAS_WARPS = 4;
constexpr int THREADS = 64 + 32 * (N_EPILOGUE_WARPS + N_BIAS_WARPS);
constexpr int OUT_STAGE_BYTES = N_EPILOGUE_WARPS * 4096, BIAS_BYTES = 32 * 32 * 4;     // 32 x 32 outputs per warp; 32 row groups x 32 columns

struct Prep {
    FusedT1Params base;
    uint16_t* za[FUSED_MAX_LAYERS];      // [planes][B][pitch_z]
    uint16_t* aa[FUSED_MAX_LAYERS];      // [planes][B][pitch_a], fp32 models
    int pitch_z[FUSED_MAX_LAYERS], pitch_a[FUSED_MAX_LAYERS];
};

template <int PLANES> struct Cfg {
    static constexpr int BK = PLANES == 1 ? 64 : 32;               // rows per stage
    static constexpr int CHUNK_BYTES = BK * 128;                   // one TMA box: BK rows x 64 columns
    static constexpr int SIDE_BYTES = 2 * CHUNK_BYTES;             // 128 columns of a plane
    static constexpr int STAGE_BYTES = 2 * PLANES * SIDE_BYTES;    // 32 KB, 48 KB
    static constexpr int STAGES = 144 * 1024 / STAGE_BYTES;        // 4, 3
    static constexpr int WINDOW = PLANES == 1 ? 12 : 4;            // stages between two drains of an accumulator: 48 additions
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 256 + OUT_STAGE_BYTES + BIAS_BYTES + 1024;
};

__device__ __forceinline__ float4 unraw4(float4 v) { return v; }
__device__ __forceinline__ float4 unraw4(uint2 r) {
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u), __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xFFFF0000u));
}
// The lane's part of a row's chunk: four elements from column c0 + 128 u + 4 lane on, zeros from column n on.  All loads stand
// before the first use of a value (with a branch a unit they went out one round trip after the other).
template <typename T>
__device__ __forceinline__ void load_chunk(const T* row, int c0, int n, bool vec, int lane, float4 (&v)[CHUNK / 128]) {
    constexpr int U = CHUNK / 128;
    if (vec) {
        typename f1::Raw4<T>::type r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + 128 * u + 4 * lane;
            r[u] = typename f1::Raw4<T>::type{};
            if (c + 4 <= n) r[u] = f1::load_raw4(row + c);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = unraw4(r[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int c = c0 + 128 * u + 4 * lane;
        if (vec && (c + 4 <= n || c >= n)) continue;          // the row's last elements, or a row without vector loads
        v[u].x = c < n ? to_f32(row[c]) : 0.f; v[u].y = c + 1 < n ? to_f32(row[c + 1]) : 0.f;
        v[u].z = c + 2 < n ? to_f32(row[c + 2]) : 0.f; v[u].w = c + 3 < n ? to_f32(row[c + 3]) : 0.f;
    }
}
template <int PLANES>
__device__ __forceinline__ void store_planes(uint16_t* dst, size_t plane, float4 v) {
    if (PLANES == 1) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    } else {
        float r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint32_t w[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const uint32_t lo = __float_as_uint(r[2 * u]), hi = __float_as_uint(r[2 * u + 1]);
                w[u] = __byte_perm(lo, hi, 0x7632);
                r[2 * u] -= __uint_as_float(lo & 0xFFFF0000u);
                r[2 * u + 1] -= __uint_as_float(hi & 0xFFFF0000u);
            }
            *reinterpret_cast<uint2*>(dst + k * plane) = make_uint2(w[0], w[1]);
        }
    }
}
}  // namespace t1p

template <typename T, int PREP_WARPS>
__global__ void __launch_bounds__(32 * PREP_WARPS)
t1_prepare_kernel(const __grid_constant__ t1p::Prep q) {
    using namespace t1p;
    constexpr int PLANES = sizeof(T) == 4 ? 3 : 1, U = CHUNK / 128;
    __shared__ float part[2 * FUSED_MAX_LAYERS][PREP_WARPS];
    __shared__ float factor_s;
    griddep_wait();
    griddep_launch_dependents();
    const FusedT1Params& p = q.base;
    const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    static_assert(2 * FUSED_MAX_LAYERS <= 32, "one store a thread");
    if (threadIdx.x < 2 * FUSED_MAX_LAYERS * PREP_WARPS) (&part[0][0])[threadIdx.x] = 0.f;
    __syncthreads();
    // rows in chunks, dealt to the warps; a warp adds up what it has of each row, in order.  all: also the rows of A, whose planes need
    // no factor
    auto chunks = [&](auto&& take) {
        int next = warp;                                          // this warp's next chunk, counted through all rows
        int begin = 0;
        for (int s = 0; s < 2 * p.L; ++s) {
            const FusedT1Layer& y = p.layer[s >> 1];
            const int n = (s & 1) ? y.d_out : y.d_in, count = (n + CHUNK - 1) / CHUNK;
            for (; next < begin + count; next += PREP_WARPS) take(s, (next - begin) * CHUNK);
            begin += count;
        }
    };
    chunks([&](int s, int c0) {
        const FusedT1Layer& y = p.layer[s >> 1];
        const bool z = s & 1;
        const int n = z ? y.d_out : y.d_in;
        const T* row = z ? static_cast<const T*>(y.Z) + (size_t)i * y.ldz : static_cast<const T*>(y.A) + (size_t)i * y.lda;
        float4 v[U];
        load_chunk(row, c0, n, (z ? y.vec_z : y.vec_a) != 0, lane, v);
        float sum = 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u) sum += (v[u].x * v[u].x + v[u].y * v[u].y) + (v[u].z * v[u].z + v[u].w * v[u].w);
        sum = warp_sum(sum);
        if (lane == 0) part[s][warp] += sum;
        if (PLANES == 3 && !z) {
            const int pitch = q.pitch_a[s >> 1];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = c0 + 128 * u + 4 * lane;
                if (c < n) store_planes<PLANES>(q.aa[s >> 1] + (size_t)i * pitch + c, (size_t)p.B * pitch, v[u]);
            }
        }
    });
    __syncthreads();
    if (warp == 0) {
        float sq = 0.f;
        if (lane < p.L) {
            float sa = 0.f, sz = 0.f;
#pragma unroll
            for (int w = 0; w < PREP_WARPS; ++w) { sa += part[2 * lane][w]; sz += part[2 * lane + 1][w]; }
            sq = (sa + (p.layer[lane].has_bias ? 1.f : 0.f)) * sz;
            p.sq[(size_t)p.layer[lane].index * p.B + i] = sq;
        }
        float total = 0.f;
        for (int l = 0; l < p.L; ++l) total += __shfl_sync(0xFFFFFFFFu, sq, l);
        if (lane == 0) {
            const float n = sqrtf(total);
            const float c = n > p.C ? p.C / n : 1.0f;
            p.clip[i] = c;
            if (p.norms) p.norms[i] = n;
            factor_s = c;
        }
    }
    __syncthreads();
    const float c = factor_s;
    chunks([&](int s, int c0) {
        if (!(s & 1)) return;
        const FusedT1Layer& y = p.layer[s >> 1];
        const T* row = static_cast<const T*>(y.Z) + (size_t)i * y.ldz;
        const int pitch = q.pitch_z[s >> 1];
        float4 v[U];
        load_chunk(row, c0, y.d_out, y.vec_z != 0, lane, v);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int col = c0 + 128 * u + 4 * lane;
            if (col < y.d_out)
                store_planes<PLANES>(q.za[s >> 1] + (size_t)i * pitch + col, (size_t)p.B * pitch,
                                     make_float4(v[u].x * c, v[u].y * c, v[u].z * c, v[u].w * c));
        }
    });
}

// 3-D tiled load: columns, rows, plane
__device__ __forceinline__ void tma_load_3d(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}

template <typename T, bool QUADS>
__global__ void __launch_bounds__(t1p::THREADS, 1)
t1_planes_kernel(const __grid_constant__ f1::Params q) {
    using namespace t1p;
    using f1::philox_normal;
    constexpr int PLANES = sizeof(T) == 4 ? 3 : 1;
    using C = Cfg<PLANES>;
    constexpr int STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES, BK = C::BK, FLUSH = C::WINDOW, CHUNK_BYTES = C::CHUNK_BYTES;
    const FusedT1Params& p = q.base;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // 1024-byte aligned, by an offset
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);             // TMA landed
    uint64_t* empty = full + STAGES;                                             // MMA done with the stage
    uint64_t* acc_full = empty + STAGES;
    uint64_t* acc_empty = acc_full + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    float4* out_stage = reinterpret_cast<float4*>(smem + STAGES * STAGE_BYTES + 256);
    float* bias_s = reinterpret_cast<float*>(smem + STAGES * STAGE_BYTES + 256 + OUT_STAGE_BYTES);     // [32][32]
    static_assert((2 * STAGES + 4) * 8 + 8 <= 256, "barrier area");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], N_EPILOGUE_WARPS); }
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0 && lane < p.L) { tma_prefetch_desc(&q.map_a[lane]); tma_prefetch_desc(&q.map_z[lane]); }
    if (warp == 1) { tmem_alloc(tmem_slot, 256); tmem_relinquish(); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    const int nkb = (p.B + BK - 1) / BK;

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            griddep_wait();                                 // planes of the launch before
            int stage = 0; uint32_t phase = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < q.total_items && ok; item += gridDim.x) {
                const Item w = decode(q, item);
                const CUtensorMap* ma = &q.map_a[w.l];
                const CUtensorMap* mz = &q.map_z[w.l];
                for (int kb = 0; kb < nkb; ++kb) {
                    ok = mbar_wait(&empty[stage], phase ^ 1, abort_flag, q.status);
                    if (!ok) break;
                    uint8_t* dst = smem + stage * STAGE_BYTES;
                    mbar_arrive_expect_tx(&full[stage], STAGE_BYTES);
#pragma unroll
                    for (int k = 0; k < PLANES; ++k)
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            tma_load_3d(dst + k * C::SIDE_BYTES + c * CHUNK_BYTES, mz, &full[stage], w.m0 + c * 64, kb * BK, k);
                            tma_load_3d(dst + (PLANES + k) * C::SIDE_BYTES + c * CHUNK_BYTES, ma, &full[stage], w.n0 + c * 64, kb * BK, k);
                        }
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc = make_idesc_bf16(BM, BN, 1, 1);
            constexpr int PRODUCTS = PLANES == 1 ? 1 : 6;
            constexpr int PZ[6] = {PLANES == 1 ? 0 : 2, 0, 1, 1, 0, 0}, PA[6] = {0, 2, 1, 0, 1, 0};      // small ones first
            int stage = 0; uint32_t phase = 0; int it = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < q.total_items && ok; item += gridDim.x) {
                uint32_t d_tmem = tmem_base;
                int buf = 0;
                for (int kb = 0; kb < nkb; ++kb) {
                    const bool window_start = (kb % FLUSH) == 0;
                    if (window_start) {
                        buf = it % NBUF;
                        ok = mbar_wait(&acc_empty[buf], ((it / NBUF) & 1) ^ 1, abort_flag, q.status);
                        if (!ok) break;
                        tc_fence_after_sync();
                        d_tmem = tmem_base + buf * BN;
                    }
                    ok = mbar_wait(&full[stage], phase, abort_flag, q.status);
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t base = smem_u32(smem + stage * STAGE_BYTES);
#pragma unroll
                    for (int k16 = 0; k16 < BK / 16; ++k16) {
                        // MN-major, 128-byte swizzle: 64-column chunks CHUNK_BYTES apart, 8-row groups 1024 bytes apart
#pragma unroll
                        for (int x = 0; x < PRODUCTS; ++x)
                            mma_bf16_ss(d_tmem, make_smem_desc_sw128(base + PZ[x] * C::SIDE_BYTES + k16 * 2048, CHUNK_BYTES, 1024),
                                        make_smem_desc_sw128(base + (PLANES + PA[x]) * C::SIDE_BYTES + k16 * 2048, CHUNK_BYTES, 1024),
                                        idesc, (window_start && k16 == 0 && x == 0) ? 0u : 1u);
                    }
                    mma_commit(&empty[stage]);
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                    if ((kb % FLUSH) == FLUSH - 1 || kb == nkb - 1) { mma_commit(&acc_full[buf]); ++it; }
                }
            }
        }
    } else if (warp >= 2 + N_EPILOGUE_WARPS) {
        // ------------------------------------------------ bias: column sums of c * zb in fp32, 32 columns of a layer at a time, dealt
        // to the CTAs.  Thread = 8 columns on rows rg, rg + 32, ... (128 columns at a time on the CTA of a tile row's first tile, a
        // thread took B / 8 rows: 25 us of loads one after the other at B = 512, the longest chain of the launch)
        griddep_wait();                                     // factors
        const int t = threadIdx.x - 64 - 32 * N_EPILOGUE_WARPS, cu = t & 3, rg = t >> 2;
        for (int unit = blockIdx.x; ; unit += gridDim.x) {
            int l = 0, u = unit;
            for (; l < p.L; ++l) {
                const int n = p.layer[l].has_bias ? (p.layer[l].d_out + 31) >> 5 : 0;
                if (u < n) break;
                u -= n;
            }
            if (l == p.L) break;
            const FusedT1Layer& y = p.layer[l];
            const T* Z = static_cast<const T*>(y.Z);
            const int m0 = u * 32, c0 = m0 + cu * 8;
            float cs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            constexpr int UNR = 8;
            if (y.vec_z && y.d_out % 4 == 0) {
                for (int r0 = rg; r0 < p.B; r0 += 32 * UNR) {         // eight rows in flight
                    typename f1::Raw4<T>::type a[UNR], b[UNR];
                    float f[UNR];
#pragma unroll
                    for (int k = 0; k < UNR; ++k) {
                        const int r = r0 + 32 * k;
                        a[k] = b[k] = typename f1::Raw4<T>::type{};
                        f[k] = 0.f;
                        if (r < p.B) f[k] = __ldcg(p.clip + r);
                        if (r < p.B && c0 + 4 <= y.d_out) a[k] = f1::load_raw4(Z + (size_t)r * y.ldz + c0);
                        if (r < p.B && c0 + 8 <= y.d_out) b[k] = f1::load_raw4(Z + (size_t)r * y.ldz + c0 + 4);
                    }
#pragma unroll
                    for (int k = 0; k < UNR; ++k) {
                        const float4 x = unraw4(a[k]), z = unraw4(b[k]);
                        cs[0] = fmaf(f[k], x.x, cs[0]); cs[1] = fmaf(f[k], x.y, cs[1]); cs[2] = fmaf(f[k], x.z, cs[2]); cs[3] = fmaf(f[k], x.w, cs[3]);
                        cs[4] = fmaf(f[k], z.x, cs[4]); cs[5] = fmaf(f[k], z.y, cs[5]); cs[6] = fmaf(f[k], z.z, cs[6]); cs[7] = fmaf(f[k], z.w, cs[7]);
                    }
                }
            } else if (y.d_out - m0 <= 16) {
                // a head of few outputs whose rows take no vector loads: thread = one column on every (128 / columns)-th row, sixteen
                // rows in flight.  (Eight columns a thread as below: two of four threads had any, and each 64 rows of eight loads at B =
                // 2048, one round trip after the other: 784-1000-1000-10 in bf16, 49 us of the second launch instead of 21.)
                const int w = y.d_out - m0, rows = 32 * N_BIAS_WARPS / w, r1 = t / w, c1 = t - r1 * w;
                float c = 0.f;
                constexpr int UNR1 = 16;
                if (r1 < rows)
                    for (int r0 = r1; r0 < p.B; r0 += rows * UNR1) {
                        T x[UNR1];
                        float f[UNR1];
#pragma unroll
                        for (int k = 0; k < UNR1; ++k) {
                            const int r = r0 + rows * k;
                            x[k] = T(0.f); f[k] = 0.f;
                            if (r < p.B) { f[k] = __ldcg(p.clip + r); x[k] = Z[(size_t)r * y.ldz + m0 + c1]; }
                        }
#pragma unroll
                        for (int k = 0; k < UNR1; ++k) c = fmaf(f[k], to_f32(x[k]), c);
                    }
                // the rows' sums in order: eight groups, then one
                bias_s[t] = c;
                f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
                c = 0.f;
                if (t < 8 * w) for (int r = r1; r < rows; r += 8) c += bias_s[r * w + c1];
                f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
                bias_s[t] = c;
                f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
                if (t < w) {
                    c = 0.f;
#pragma unroll
                    for (int g = 0; g < 8; ++g) c += bias_s[g * w + t];
                    const int m = m0 + t;
                    if (p.noise_scale > 0.f) c = fmaf(p.noise_scale, philox_normal((size_t)m, p.stream_id0 + 2ull * y.index + 1, p.k0, p.k1), c);
                    y.gb[m] = c;
                }
                f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
                continue;
            } else if (c0 < y.d_out) {
                constexpr int ROWS = 4;
                for (int r0 = rg; r0 < p.B; r0 += 32 * ROWS) {
                    T x[ROWS][8];
                    float f[ROWS];
#pragma unroll
                    for (int k = 0; k < ROWS; ++k) {
                        const int r = r0 + 32 * k;
                        f[k] = 0.f;
                        if (r < p.B) f[k] = __ldcg(p.clip + r);
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            x[k][j] = T(0.f);
                            if (r < p.B && c0 + j < y.d_out) x[k][j] = Z[(size_t)r * y.ldz + c0 + j];
                        }
                    }
#pragma unroll
                    for (int k = 0; k < ROWS; ++k)
#pragma unroll
                        for (int j = 0; j < 8; ++j) cs[j] = fmaf(f[k], to_f32(x[k][j]), cs[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) bias_s[rg * 32 + cu * 8 + j] = cs[j];
            f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
            float c = 0.f;
#pragma unroll
            for (int g = 0; g < 8; ++g) c += bias_s[((t >> 5) * 8 + g) * 32 + lane];
            f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
            bias_s[t] = c;
            f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
            if (t < 32 && m0 + t < y.d_out) {
                c = (bias_s[t] + bias_s[32 + t]) + (bias_s[64 + t] + bias_s[96 + t]);
                const int m = m0 + t;
                if (p.noise_scale > 0.f) c = fmaf(p.noise_scale, philox_normal((size_t)m, p.stream_id0 + 2ull * y.index + 1, p.k0, p.k1), c);
                y.gb[m] = c;
            }
            f1::named_barrier_sync(1, 32 * N_BIAS_WARPS);
        }
    } else {
        // ------------------------------------------------ epilogue (16 warps)
        // Warp w may touch tensor-memory lanes 32*(w % 4) .. +31; the four warps of a lane quarter take 32 columns each.  Thread = one
        // output row.  Sixteen warps for the noise: with eight the generator of a wide model's 21 million outputs set the pace.
        const int quarter = warp & 3, ew = warp - 2, g = ew >> 2;
        int it = 0;
        bool ok = true;
        float4* st = out_stage + ew * 256;
        for (int item = blockIdx.x; item < q.total_items && ok; item += gridDim.x) {
            const Item w = decode(q, item);
            const FusedT1Layer& y = p.layer[w.l];
            const unsigned long long sid_w = p.stream_id0 + 2ull * y.index;
            const uint32_t s0 = (uint32_t)sid_w, s1 = (uint32_t)(sid_w >> 32);
            const int m_base = w.m0 + quarter * 32, n_base = w.n0 + g * 32;
            // accumulators start from the noise of their outputs, drawn while the MMAs run
            float acc[32];
            const size_t e_row = (size_t)(m_base + lane) * y.d_in;
            const bool draw = p.noise_scale > 0.f && m_base + lane < y.d_out && n_base < y.d_in;
            if (!__any_sync(0xFFFFFFFFu, draw)) {
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[j] = 0.f;
            } else if (QUADS) {
                // straight-line code, four independent Philox blocks at a time
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float z[4][4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) normals_block((e_row + n_base + 16 * h + 4 * k) >> 2, s0, s1, p.k0, p.k1, z[k]);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int u = 0; u < 4; ++u) acc[16 * h + 4 * k + u] = draw ? p.noise_scale * z[k][u] : 0.f;
                }
            } else {
                // some layer's rows start inside a Philox block: a group of four outputs takes parts of two blocks
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[j] = 0.f;
#pragma unroll 1
                for (int k = 0; k < 8; ++k) {
                    float z[4];
                    normals_at(e_row + n_base + 4 * k, s0, s1, p.k0, p.k1, z);
#pragma unroll
                    for (int j = 0; j < 32; ++j) acc[j] = (j >> 2) == k && draw ? p.noise_scale * z[j & 3] : acc[j];
                }
            }
            for (int kb = 0; kb < nkb; kb += FLUSH, ++it) {
                const int buf = it % NBUF;
                ok = mbar_wait(&acc_full[buf], (it / NBUF) & 1, abort_flag, q.status);
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * BN + g * 32;
                uint32_t v[2][16];
                tmem_ld_32x16(t_row, v[0]);
                tmem_ld_32x16(t_row + 16, v[1]);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[j] += __uint_as_float(v[j >> 4][j & 15]);
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[buf]);
            }
            if (!ok) break;
            // the 32 x 32 block through shared memory: every store then covers 4 rows x 128 bytes, whole lines (16 rows x 32 bytes,
            // four times the requests to L2: 57 us instead of 50 on the wide model, before the loads of the bias sums were mended)
#pragma unroll
            for (int j = 0; j < 8; ++j)
                st[lane * 8 + (j ^ (lane & 7))] = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
            __syncwarp();
            const int jj = lane & 7, n = n_base + 4 * jj;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int rr = 4 * i + (lane >> 3);
                const float4 x = st[rr * 8 + (jj ^ (rr & 7))];
                if (m_base + rr < y.d_out && n < y.d_in) {
                    float* dst = y.gW + (size_t)(m_base + rr) * y.d_in + n;
                    if (QUADS) {
                        *reinterpret_cast<float4*>(dst) = x;
                    } else {
                        const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                        for (int u = 0; u < 4; ++u) if (n + u < y.d_in) dst[u] = xs[u];
                    }
                }
            }
            __syncwarp();
        }
    }

    // ---------------------------------------------------- teardown
    if (*abort_flag) {
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) { tc_fence_after_sync(); tmem_dealloc(tmem_base, 256); }
}

}  // namespace tc
}  // namespace dpclip
