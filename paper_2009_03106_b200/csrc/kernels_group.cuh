// Zb^T diag(f) A of MANY layers in one launch, on CTA pairs (tcgen05.mma.cta_group::2): the per-example norms by the
// materialised product and the clipped sums of fp32 layers.
//
// Why one launch.  A small model's layers are each a chain of latencies (set-up, first loads, drain) that fills few
// SMs, and launched one after the other they add up: seven fp32 layers of 148 to 592 features (B = 61, T = 48) were 7
// norm launches of 10 to 20 us and 14 clipped-sum launches, 252 us a step for 1.1 GFLOP.  Here the layers' work is one sequence
// of units cut into equal shares, one per CTA pair.
//
// Why pairs.  What bounds the fp32 product is the shared-memory port: an fp32 operand tile is written by TMA, read and
// split into planes, and the planes are read several times by the MMAs.  On one CTA with a 128 x 128 tile that was 208 KB
// per 32 rows for 768 clocks of MMAs (47 % at best, 36 % measured).  A pair on a 256 x 256 tile needs the same 208 KB in
// each CTA for twice the MMA work: every CTA holds 128 columns of the M side and half of the N side.
//
// Tile.  The M side (256 columns of one operand, 128 per CTA) is A or Zb, whichever wastes less padding; the N side is
// N = 64, 128, 192 or 256 columns of the other, N/2 per CTA.
//
// Work.  GRAD: unit = one stage (BK rows) of one tile; layer after layer, tile after tile; pair r takes the units
//              [run_begin[r], run_begin[r + 1]), cut so that every run costs the same.  A run may end in the middle of a
//              tile: each (tile, run) leaves one partial tile in slot tile + r of the workspace (tile and r both only
//              grow along the sequence, so no slot is used twice), and reduce_group_kernel adds a tile's slots in order.
//       NORM: unit = one (example, tile); runs end between units; squares are summed into sq with atomics.
//
// Numbers.      fp32 inputs: x = b0 + b1 + b2, three bf16 terms cut off the top of the fp32 word: 3 x 8 bits, exact.  Six products,
//                         b0 b0, b0 b1, b1 b0, b1 b1, b0 b2, b2 b0; what is dropped (b1 b2, b2 b1) is below 2^-21 of a
//                         product, 2^-24 on average, always toward zero.  The tensor core needs as long for them as for three tf32 products (which drop as much),
//                         but 16-bit operands come out of the MN-major layout at full rate: the twelve tf32 MMAs of a 256 x
//                         256 stage took 1.2 us where 0.8 is nominal.
//                         The tensor core's accumulation truncates, a bias toward zero that grows with the number of additions:
//                         the five small products go to an accumulator of their own, so that the large one sees two additions
//                         a stage instead of twelve, and every FLUSH stages (48 additions) both are added up outside.  (Draining
//                         one accumulator every four stages into registers of the warps that also prepare the stages took 2 us
//                         each time, a quarter of the kernel.)
//
// Measured (fp32): the loop of 256 x 256 tiles takes 1.15 us a stage, 1.6 PFLOP/s of bf16 products, the tensor core's rate
// (two plane stages and four raw ones, or three and two: the same).  Seven layers of 512 and 2048 features, B = 32, T = 128:
// norms 159 us, clipped sums 171 us, reduce 28 us, where one launch per layer took 305, 310 and 38.  Of those the loop is 127
// us each (8192 stages on 74 pairs; tensor pipe active 56 and 54 % of a launch under ncu, when the norms took 172); the norms lose the rest to
// the drain behind the four stages of an example, the sums to fill, drains and partial tiles.
//
// Roles: warp 0 TMA (each CTA its own operands, plain loads), warp 1 MMA issuer (rank 0), 16 warps that prepare every
// stage (factor, planes, bias column sums), 8 epilogue warps that take the finished accumulators.
// Barriers as in zta_pair_kernel; every wait is bounded.
#pragma once
#include "kernels_tc_pair.cuh"

namespace dpclip {
namespace tc {
namespace zg {
constexpr int BM = 256, BM_CTA = 128, BN_MAX = 256;
constexpr int PITCH = 256;                           // fp32 elements between two N-side columns of a partial tile
constexpr size_t SLOT_ELEMS = (size_t)BN_MAX * PITCH;
constexpr int PREP = 16, EPI = 8, THREADS = 64 + 32 * (PREP + EPI);
constexpr int MAX_LAYERS = 16, MAX_RUNS = kNumSMs / 2;
constexpr int FLUSH = 24;                            // stages between two drains of a tile's accumulators ...
constexpr int FLUSH_ONE = 4;                         // ... and in a segment of at most so many, one accumulator takes all products

// A stage = BK rows.  TMA fills a ring of raw stages, the planes of a stage are written into a second ring.
struct Cfg {
    static constexpr int BK = 32;                                  // rows per stage
    static constexpr int BOX = 32;                                 // columns per TMA box (128 bytes)
    static constexpr int BOX_BYTES = BK * 128;
    static constexpr int RAW_SIDE = (BM_CTA / BOX) * BOX_BYTES;    // 128 columns as loaded: 16 KB
    static constexpr int CHUNK_BYTES = BK * 128;                   // 64 bf16 columns of an operand plane
    static constexpr int SIDE_BYTES = 2 * CHUNK_BYTES;             // 128 columns of a plane: 8 KB
    static constexpr int PLANES = 3;
    static constexpr int OFF_M = 0, OFF_N = PLANES * SIDE_BYTES;
    static constexpr int STAGE_BYTES = 2 * PLANES * SIDE_BYTES, STAGES = 2;
    static constexpr int OFF_RAW = STAGES * STAGE_BYTES;           // raw ring behind the planes
    static constexpr int RAW_BYTES = 2 * RAW_SIDE, RAW_STAGES = 4;
    static constexpr int RING_BYTES = STAGES * STAGE_BYTES + RAW_STAGES * RAW_BYTES;
    static constexpr int SMEM_BYTES = RING_BYTES + 256 + 1024;
};

// Eight fp32 values as three bf16 terms each (packed in pairs), every term the top 16 bits of what the ones before left.
__device__ __forceinline__ void split_bf16x3(const float (&x)[8], uint4 (&b)[3]) {
    uint32_t* w[3] = {reinterpret_cast<uint32_t*>(&b[0]), reinterpret_cast<uint32_t*>(&b[1]), reinterpret_cast<uint32_t*>(&b[2])};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        float r0 = x[2 * u], r1 = x[2 * u + 1];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t v0 = __float_as_uint(r0), v1 = __float_as_uint(r1);
            w[k][u] = __byte_perm(v0, v1, 0x7632);
            r0 -= __uint_as_float(v0 & 0xFFFF0000u);
            r1 -= __uint_as_float(v1 & 0xFFFF0000u);
        }
    }
}

struct Layer {
    int T, R;                      // rows per example, rows in all
    int d_m, d_n, z_on_m;          // widths of the M and N side; 1: the M side is Zb, 0: it is A
    int tiles_m, tiles_n, N;       // N = tile width of the N side
    int nkb;                       // stages of a tile (GRAD) or of an item (NORM)
    int tile0, tiles;              // GRAD: the launch covers tiles tile0 .. tile0 + tiles - 1 of the layer
    int tile_base, unit_base;      // first tile / first unit of the layer in the launch
    int do_bias;
    const float* clip;             // GRAD: [B] or NULL
    float* gW; float* gb; long ldg; int vec_ok;
    float* sq;                     // NORM: [B]
    uint32_t sw0, sw1, sb0, sb1;   // noise streams
    int blk_begin;                 // reduce: first 32 x 32 block of the layer
};
struct Params {
    int n_layers, n_runs;
    int run_begin[MAX_RUNS + 1];
    float* part; float* bias_part; // [slots][256][PITCH], [slots][256]
    int n_slots;
    int* status;
    float noise_scale; uint32_t k0, k1;
    gram::FactorsTail tail;
    Layer layer[MAX_LAYERS];
    int n_blocks;                  // reduce
    // a layer whose partial tiles do not fit the workspace at once goes chunk of tiles by chunk of tiles; its bias sums add
    // up over the chunks
    int first_chunk, last_chunk;
};
struct Maps { CUtensorMap m[MAX_LAYERS], n[MAX_LAYERS]; };

// Tensor memory is two slots of 256 columns.  A window takes one of them in turn -- the large products in the first N
// columns, the small ones 128 further -- or, with N > 128, both: the large products in slot 0, the small ones in 1, and
// the next window waits for its drain.  A segment of at most FLUSH_ONE stages (48 additions in all) keeps everything in one
// accumulator of one slot: the drain, 1.5 us of the 6 us of such an item at N = 256, then runs beside the next one's MMAs.
// Every role walks the same sequence.
struct AccRing {
    uint32_t uses0 = 0, uses1 = 0, next = 0;
    bool wide = false; uint32_t slot = 0;
    __device__ __forceinline__ void take(bool w) {
        wide = w;
        slot = w ? 0 : next;
        if (!w) next ^= 1;
    }
    __device__ __forceinline__ uint32_t uses(uint32_t s) const { return s ? uses1 : uses0; }       // of a slot, before this one
    __device__ __forceinline__ void done() {
        if (wide || slot == 0) ++uses0;
        if (wide || slot == 1) ++uses1;
    }
};

struct Seg { int layer, tm, tn, kb0, kb1, row0, row_end, example, slot, units; };

template <bool NORM>
__device__ __forceinline__ Seg segment_at(const Params& p, int u, int u_end, int run) {
    Seg s;
    int l = 0;
#pragma unroll 1
    while (l + 1 < p.n_layers && u >= p.layer[l + 1].unit_base) ++l;
    const Layer& y = p.layer[l];
    const int local = u - y.unit_base;
    s.layer = l;
    int tile;
    if (NORM) {
        s.example = local / y.tiles;
        tile = local - s.example * y.tiles;
        s.kb0 = 0; s.kb1 = y.nkb;
        s.row0 = s.example * y.T; s.row_end = s.row0 + y.T;
        s.units = 1; s.slot = run;
    } else {
        const int t = local / y.nkb;
        s.kb0 = local - t * y.nkb;
        s.kb1 = min(y.nkb, s.kb0 + (u_end - u));
        s.units = s.kb1 - s.kb0;
        s.row0 = 0; s.row_end = y.R; s.example = 0;
        s.slot = y.tile_base + t + run;
        tile = y.tile0 + t;
    }
    s.tm = tile / y.tiles_n; s.tn = tile - s.tm * y.tiles_n;
    return s;
}
}  // namespace zg

template <bool NORM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(zg::THREADS, 1)
zta_group_kernel(const __grid_constant__ zg::Maps maps, const __grid_constant__ zg::Params p) {
    using namespace zg;
    using C = Cfg;
    constexpr int STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES, BK = C::BK, CHUNK_BYTES = C::CHUNK_BYTES;
    constexpr int RAW_STAGES = C::RAW_STAGES;
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned by an OFFSET from the array (keeps the accesses in the shared state space), the same in both CTAs
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::RING_BYTES);          // [RAW_STAGES] TMA landed (this CTA)
    uint64_t* raw_free = full + RAW_STAGES;                                      // [RAW_STAGES] raw stage read (own)
    uint64_t* ready = raw_free + RAW_STAGES;                                     // stage prepared (rank 0's is used)
    uint64_t* empty = ready + STAGES;                                            // MMAs done with the stage (each CTA's own)
    uint64_t* acc_full = empty + STAGES;                                         // [2] accumulator complete (each CTA's own)
    uint64_t* acc_empty = acc_full + 2;                                          // [2] accumulator drained (rank 0's is used)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    static_assert((2 * RAW_STAGES + 2 * STAGES + 4) * 8 + 8 <= 256, "barrier area");
    static_assert(C::SMEM_BYTES <= 227 * 1024, "shared memory");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();                  // 0 = issues the MMAs
    const int run = blockIdx.x >> 1;
    const int u_begin = p.run_begin[run], u_end = p.run_begin[run + 1];
    if (threadIdx.x == 0) {
        for (int s = 0; s < RAW_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&raw_free[s], PREP); }
        for (int s = 0; s < STAGES; ++s) { mbar_init(&ready[s], 2 * PREP); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * EPI); }
        *abort_flag = 0;
        mbar_fence_init();
        for (int l = 0; l < p.n_layers; ++l) { tma_prefetch_desc(&maps.m[l]); tma_prefetch_desc(&maps.n[l]); }
    }
    if (warp == 1) { tmem_alloc_pair(tmem_slot, 512); tmem_relinquish_pair(); }
    tc_fence_before_sync();
    cluster_sync_all();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Norms may follow the launch that copies their operands, clipped sums the one that computes the factors: of the latter the loads
    // run ahead, and whoever passes the launch on (warp 1) waits in either.
    if (NORM || warp >= 1) griddep_wait();

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            int stage = 0; uint32_t phase = 0;
            bool ok = true;
            [[maybe_unused]] int tr = 0;
            for (int u = u_begin; u < u_end && ok;) {
                const Seg w = segment_at<NORM>(p, u, u_end, run);
                const Layer& y = p.layer[w.layer];
                const CUtensorMap* map_m = &maps.m[w.layer];
                const CUtensorMap* map_n = &maps.n[w.layer];
                const int xm = w.tm * BM + (int)rank * BM_CTA, half = y.N >> 1, xn = w.tn * y.N + (int)rank * half;
                const int n_boxes = (half + C::BOX - 1) / C::BOX;
                for (int kb = w.kb0; kb < w.kb1; ++kb) {
                    ok = mbar_wait(&raw_free[stage], phase ^ 1, abort_flag, p.status);
                    if (!ok) break;
                    DPCLIP_TRACE_AT(0, tr); ++tr;
                    uint8_t* dst = smem + C::OFF_RAW + stage * C::RAW_BYTES;
                    const int r = w.row0 + kb * BK;
                    mbar_arrive_expect_tx(&full[stage], C::RAW_SIDE + n_boxes * C::BOX_BYTES);
#pragma unroll
                    for (int c = 0; c < BM_CTA / C::BOX; ++c)
                        tma_load_2d(dst + c * C::BOX_BYTES, map_m, &full[stage], xm + c * C::BOX, r);
#pragma unroll 1
                    for (int c = 0; c < n_boxes; ++c)
                        tma_load_2d(dst + C::RAW_SIDE + c * C::BOX_BYTES, map_n, &full[stage], xn + c * C::BOX, r);
                    if (++stage == RAW_STAGES) { stage = 0; phase ^= 1; }
                }
                u += w.units;
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer (rank 0 only)
        if (lane == 0 && rank != 0) griddep_launch_dependents();
        if (lane == 0 && rank == 0) {
            int stage = 0; uint32_t phase = 0;
            AccRing ring;
            bool ok = true;
            [[maybe_unused]] int tr = 0;
            for (int u = u_begin; u < u_end && ok;) {
                const Seg w = segment_at<NORM>(p, u, u_end, run);
                const Layer& y = p.layer[w.layer];
                const uint32_t idesc = make_idesc_bf16(BM, y.N, 1, 1);
                const bool two = w.kb1 - w.kb0 > FLUSH_ONE;
                uint32_t d_tmem = tmem_base, d_small = tmem_base;
                for (int kb = w.kb0; kb < w.kb1; ++kb) {
                    const int k = kb - w.kb0;
                    const bool start = (k % FLUSH) == 0;
                    if (start) {
                        ring.take(two && y.N > 128);
                        ok = mbar_wait(&acc_empty[ring.slot], (ring.uses(ring.slot) & 1) ^ 1, abort_flag, p.status) &&
                             (!ring.wide || mbar_wait(&acc_empty[1], (ring.uses(1) & 1) ^ 1, abort_flag, p.status));
                        if (!ok) break;
                        tc_fence_after_sync();
                        d_tmem = tmem_base + ring.slot * 256;
                        d_small = !two ? d_tmem : d_tmem + (ring.wide ? 256 : 128);
                    }
                    ok = mbar_wait(&ready[stage], phase, abort_flag, p.status);
                    if (!ok) break;
                    DPCLIP_TRACE_AT(2, tr); ++tr;
                    tc_fence_after_sync();
                    const uint32_t base = smem_u32(smem + stage * STAGE_BYTES);
                    // MN-major, 128-byte swizzle: 64-column chunks CHUNK_BYTES apart, 8-row groups 1024 bytes apart
                    constexpr int PM[6] = {2, 0, 1, 1, 0, 0}, PN[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
                    for (int k4 = 0; k4 < BK / 16; ++k4) {
#pragma unroll
                        for (int x = 0; x < 6; ++x)
                            mma_bf16_ss_pair(x == 5 ? d_tmem : d_small,
                                             make_smem_desc_sw128(base + C::OFF_M + PM[x] * C::SIDE_BYTES + k4 * 2048, CHUNK_BYTES, 1024),
                                             make_smem_desc_sw128(base + C::OFF_N + PN[x] * C::SIDE_BYTES + k4 * 2048, CHUNK_BYTES, 1024),
                                             idesc, (start && k4 == 0 && (x == 0 || (x == 5 && two))) ? 0u : 1u);
                    }
                    mma_commit_pair(&empty[stage], 3);          // frees the stage in both CTAs
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                    if (kb == w.kb1 - 1 || (k % FLUSH) == FLUSH - 1) {
                        mma_commit_pair(&acc_full[ring.slot], 3);
                        if (ring.wide) mma_commit_pair(&acc_full[1], 3);
                        ring.done();
                    }
                }
                u += w.units;
            }
            griddep_launch_dependents();                        // the launch that follows may place its CTAs as SMs fall idle
        }
    } else if (warp < 2 + PREP) {
        // ------------------------------------------------ preparation
        // A side of a stage is 128 columns; warp wk takes 8 of them over all rows, lane = row: a column's bias sum stays inside a warp, and eight lanes' 16-byte accesses fall on different banks.  The
        // 16-byte units of a row sit where the 128-byte swizzle puts them, at the same place for all rows of a thread.
        const int wk = warp - 2;
        constexpr int NR = BK / 32;
        const uint32_t off = (wk >> 3) * CHUNK_BYTES + lane * 128 + (((wk & 7) ^ (lane & 7)) << 4);
        // the two fp32 units of those columns in a raw stage
        const uint32_t raw0 = (wk >> 2) * C::BOX_BYTES + lane * 128 + (((2 * (wk & 3)) ^ (lane & 7)) << 4);
        const uint32_t raw1 = (wk >> 2) * C::BOX_BYTES + lane * 128 + (((2 * (wk & 3) + 1) ^ (lane & 7)) << 4);
        const uint32_t ready0 = mapa_shared(smem_u32(ready), 0);
        int stage = 0; uint32_t phase = 0;
        int raw = 0; uint32_t raw_phase = 0;                   // position in the raw ring
        bool ok = true;
        [[maybe_unused]] int tr = 0;
        for (int u = u_begin; u < u_end && ok;) {
            const Seg w = segment_at<NORM>(p, u, u_end, run);
            const Layer& y = p.layer[w.layer];
            const int T = y.T, z_on_m = y.z_on_m;
            const int half = y.N >> 1;
            const bool n_live = wk * 8 < half;                 // this warp's columns exist on the N side
            const bool z_live = z_on_m || n_live;
            const float* clip = NORM ? nullptr : y.clip;
            // every tile of the other side sees the same Zb rows: GRAD deals the bias sums of stage kb to the tile with kb %
            // tiles == its index there; NORM squares them, so one tile takes them all
            const int o_tiles = z_on_m ? y.tiles_n : y.tiles_m, o_tile = z_on_m ? w.tn : w.tm;
            float cs[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) cs[j] = 0.f;
            for (int kb = w.kb0; kb < w.kb1; ++kb) {
                // factors of this stage's rows, fetched before waiting for the tile
                const int blk0 = w.row0 + kb * BK;
                float fr[NR];
                if (!NORM) {
                    const int e_first = blk0 / T, rem0 = blk0 - e_first * T;
                    const bool uniform = rem0 + BK <= T && blk0 + BK <= w.row_end;
#pragma unroll
                    for (int i = 0; i < NR; ++i) {
                        const int rl = lane + 32 * i;
                        // past the last row TMA filled zeros; the factor only has to be finite there
                        fr[i] = blk0 + rl >= w.row_end ? 0.f : !clip ? 1.f : __ldg(clip + e_first + (uniform ? 0 : (rem0 + rl) / T));
                    }
                }
                const bool bias_here = y.do_bias && z_live && (NORM ? o_tile == 0 : (kb % o_tiles) == o_tile);
                ok = mbar_wait(&full[raw], raw_phase, abort_flag, p.status);
                if (!ok) break;
                if (threadIdx.x == 64) { DPCLIP_TRACE_AT(1, tr); ++tr; }
                uint8_t* st = smem + stage * STAGE_BYTES + off;
                const uint8_t* rw = smem + C::OFF_RAW + raw * C::RAW_BYTES;
                float4 x[2][2];
#pragma unroll
                for (int side = 0; side < 2; ++side) {                   // 0: M, 1: N
                    x[side][0] = *reinterpret_cast<const float4*>(rw + side * C::RAW_SIDE + raw0);
                    x[side][1] = *reinterpret_cast<const float4*>(rw + side * C::RAW_SIDE + raw1);
                }
                if (NORM && blk0 + lane >= w.row_end) {
                    // rows of the next example are cleared on both sides: an infinity or NaN there times a factor of 0 would
                    // be this one's norm
#pragma unroll
                    for (int side = 0; side < 2; ++side) x[side][0] = x[side][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                uint4 b3[2][3];
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    if (side == 1 && !n_live) continue;
                    float v[8] = {x[side][0].x, x[side][0].y, x[side][0].z, x[side][0].w,
                                  x[side][1].x, x[side][1].y, x[side][1].z, x[side][1].w};
                    if ((side == 0) == (z_on_m != 0)) {
                        if (!NORM) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) v[k] *= fr[0];
                        }
                        if (bias_here) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) cs[k] += v[k];
                        }
                    }
                    split_bf16x3(v, b3[side]);
                }
                ok = mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.status);
                if (!ok) break;
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    if (side == 1 && !n_live) continue;
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        *reinterpret_cast<uint4*>(st + side * C::OFF_N + k * C::SIDE_BYTES) = b3[side][k];
                }
                // The raw stage is given back only here: the stores above used the values, so the loads are complete.  (Given
                // back right after the loads were issued, it was refilled under them now and then.)
                __syncwarp();
                if (lane == 0) mbar_arrive(&raw_free[raw]);
                if (++raw == RAW_STAGES) { raw = 0; raw_phase ^= 1; }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(ready0 + stage * 8);
                if (threadIdx.x == 64) { DPCLIP_TRACE_AT(1, tr); ++tr; }
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            if (!ok) break;
            if (y.do_bias && (!NORM || o_tile == 0)) {
                // a column's sum lies in one warp; a GRAD segment writes its sums whether it took any or not, so the reduce can
                // add all of a tile
                float ssq = 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float c = warp_sum(cs[j]);
                    ssq = fmaf(c, c, ssq);
                    if (!NORM && lane == 0 && z_live && DPCLIP_IN_RANGE(w.slot, p.n_slots, p.status))
                        p.bias_part[(size_t)w.slot * 256 + rank * (z_on_m ? BM_CTA : half) + wk * 8 + j] = c;
                }
                if (NORM && lane == 0 && z_live) atomicAdd(y.sq + w.example, ssq);
            }
            u += w.units;
        }
    } else {
        // ------------------------------------------------ epilogue
        // Warp w may touch tensor-memory lanes 32*(w % 4) .. +31; the two warps of a lane quarter take half of the N columns
        // each.  A tile's accumulators may come in several windows: the sums so far wait in the partial tile (NORM: the run's
        // own slot), where every thread finds what it wrote itself.
        const int quarter = warp & 3, g = (warp - 2 - PREP) >> 2;
        const uint32_t acc_empty0 = mapa_shared(smem_u32(acc_empty), 0);
        AccRing ring;
        bool ok = true;
        [[maybe_unused]] int etr = 0;
        for (int u = u_begin; u < u_end && ok;) {
            const Seg w = segment_at<NORM>(p, u, u_end, run);
            const Layer& y = p.layer[w.layer];
            const int nq = y.N >> 1;                           // columns of this warp: 32, 64, 96 or 128
            const bool in_range = DPCLIP_IN_RANGE(w.slot, p.n_slots, p.status);
            float* dst = p.part + (size_t)w.slot * SLOT_ELEMS + (size_t)(g * nq) * PITCH + rank * BM_CTA + quarter * 32 + lane;
            const int windows = (w.kb1 - w.kb0 + FLUSH - 1) / FLUSH;
            const bool two = w.kb1 - w.kb0 > FLUSH_ONE;
            float fro = 0.f;
            for (int win = 0; win < windows; ++win) {
                ring.take(two && y.N > 128);
                if (threadIdx.x == 64 + 32 * PREP) { DPCLIP_TRACE_AT(3, etr); ++etr; }
                ok = mbar_wait(&acc_full[ring.slot], ring.uses(ring.slot) & 1, abort_flag, p.status) &&
                     (!ring.wide || mbar_wait(&acc_full[1], ring.uses(1) & 1, abort_flag, p.status));
                if (!ok) break;
                if (threadIdx.x == 64 + 32 * PREP) { DPCLIP_TRACE_AT(3, etr); ++etr; }
                tc_fence_after_sync();
                const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + ring.slot * 256 + g * nq;
                const uint32_t to_small = ring.wide ? 256 : 128;
                const bool last = win == windows - 1;
                if (NORM && !two) {
                    // short examples: one window of one accumulator, only its squares are wanted.  The drain is what such an item waits
                    // for: 32 columns are under way at a time, in four chains of additions (16 in one chain: norms of 160 examples of
                    // 32 positions, 512 to 2048 features, 388 us, here 248; 59 positions 250, 209; 128 positions 163, 160)
                    float f4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                    for (int h = 0; h < nq; h += 32) {
                        uint32_t v[32];
                        tmem_ld_32x32(t_row + h, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 32; ++j) f4[j & 3] = fmaf(__uint_as_float(v[j]), __uint_as_float(v[j]), f4[j & 3]);
                    }
                    fro = (f4[0] + f4[1]) + (f4[2] + f4[3]);
                } else
#pragma unroll 1
                for (int h = 0; h < nq; h += 16) {
                    float x[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) x[j] = 0.f;
                    if (win > 0 && in_range) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) x[j] = dst[(size_t)(h + j) * PITCH];
                    }
                    uint32_t v[16];
                    tmem_ld_32x16(t_row + h, v);
                    if (two) {
                        uint32_t v2[16];
                        tmem_ld_32x16(t_row + to_small + h, v2);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) x[j] += __uint_as_float(v[j]) + __uint_as_float(v2[j]);
                    } else {
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) x[j] = __uint_as_float(v[j]);
                    }
                    if (NORM && last) {
                        // columns beyond the widths were zero-filled by TMA: they add nothing
#pragma unroll
                        for (int j = 0; j < 16; ++j) fro = fmaf(x[j], x[j], fro);
                    } else if (in_range) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) dst[(size_t)(h + j) * PITCH] = x[j];
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive_cluster(acc_empty0 + ring.slot * 8);
                    if (ring.wide) mbar_arrive_cluster(acc_empty0 + 8);
                }
                ring.done();
                if (threadIdx.x == 64 + 32 * PREP) { DPCLIP_TRACE_AT(3, etr); ++etr; }
            }
            if (!ok) break;
            if (NORM) {
                fro = warp_sum(fro);
                if (lane == 0) atomicAdd(y.sq + w.example, fro);
            }
            u += w.units;
        }
    }

    // ---------------------------------------------------- teardown
    if (*abort_flag) {
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
    tc_fence_before_sync();
    cluster_sync_all();             // nobody frees tensor memory or exits while its partner may still signal it
    if (warp == 1) { tc_fence_after_sync(); tmem_dealloc_pair(tmem_base, 512); }
    if (NORM) gram::factors_tail(p.tail);
}

// ---------------------------------------------------------------------------
// Second stage of the clipped sums: every output element = the sum of its tile's partial tiles in run order (+ noise).
// CTA = 32 x 32 outputs, thread = four consecutive elements of a row of gW.  With A on the M side a partial tile's rows
// run along d_in like gW's and are read as they lie; with Zb there the block is turned through shared memory.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
reduce_group_kernel(const __grid_constant__ zg::Params p) {
    using namespace zg;
    __shared__ float turn[32][33];
    griddep_wait();
    auto run_of = [&](int u) {                                 // last run that begins at or before unit u
        int lo = 0, hi = p.n_runs;
        while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (p.run_begin[mid] <= u) lo = mid; else hi = mid; }
        return lo;
    };
    for (int blk = blockIdx.x; blk < p.n_blocks; blk += gridDim.x) {
        int l = 0;
        while (l + 1 < p.n_layers && blk >= p.layer[l + 1].blk_begin) ++l;
        const Layer& y = p.layer[l];
        // blocks are numbered tile by tile: 8 along the M side, N / 32 along the N side
        const int per_tile = 8 * (y.N >> 5);
        const int local = blk - y.blk_begin, t = local / per_tile, r = local - t * per_tile;
        const int bm = r & 7, bn = r >> 3;
        const int tile = y.tile0 + t, tm = tile / y.tiles_n, tn = tile - tm * y.tiles_n;
        const int m0 = tm * BM + bm * 32, n0 = tn * y.N + bn * 32;
        if (m0 >= y.d_m || n0 >= y.d_n) continue;              // the same for the whole CTA
        const int u0 = y.unit_base + t * y.nkb;
        const int r0 = run_of(u0), r1 = run_of(u0 + y.nkb - 1);
        const float* src = p.part + (size_t)(y.tile_base + t + r0) * SLOT_ELEMS + (size_t)(bn * 32) * PITCH + bm * 32;
        const int row = threadIdx.x >> 3, c4 = (threadIdx.x & 7) << 2;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = r0; k <= r1; k += 4) {                    // four loads in flight
            float4 v[4];
#pragma unroll
            for (int h = 0; h < 4; ++h)
                v[h] = k + h <= r1 ? __ldcs(reinterpret_cast<const float4*>(src + (size_t)(k + h - r0) * SLOT_ELEMS + row * PITCH + c4))
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int h = 0; h < 4; ++h) { acc.x += v[h].x; acc.y += v[h].y; acc.z += v[h].z; acc.w += v[h].w; }
        }
        if (y.z_on_m) {
            __syncthreads();
            turn[c4][row] = acc.x; turn[c4 + 1][row] = acc.y; turn[c4 + 2][row] = acc.z; turn[c4 + 3][row] = acc.w;
            __syncthreads();
            acc = make_float4(turn[row][c4], turn[row][c4 + 1], turn[row][c4 + 2], turn[row][c4 + 3]);
        }
        const int o = (y.z_on_m ? m0 : n0) + row, i = (y.z_on_m ? n0 : m0) + c4;
        const int d_out = y.z_on_m ? y.d_m : y.d_n, d_in = y.z_on_m ? y.d_n : y.d_m;
        if (o >= d_out || i >= d_in) continue;
        if (p.noise_scale > 0.f) {
            float z[4];
            normals_at((size_t)o * d_in + i, y.sw0, y.sw1, p.k0, p.k1, z);
            acc.x = fmaf(p.noise_scale, z[0], acc.x); acc.y = fmaf(p.noise_scale, z[1], acc.y);
            acc.z = fmaf(p.noise_scale, z[2], acc.z); acc.w = fmaf(p.noise_scale, z[3], acc.w);
        }
        float* dst = y.gW + (size_t)o * y.ldg + i;
        if (y.vec_ok && i + 4 <= d_in) {
            *reinterpret_cast<float4*>(dst) = acc;
        } else {
            const float xs[4] = {acc.x, acc.y, acc.z, acc.w};
            for (int k = 0; k < 4; ++k)
                if (i + k < d_in) dst[k] = xs[k];
        }
    }
    // the bias sums: one warp per output, lanes over the tiles of the other side
    const int lane = threadIdx.x & 31;
    int total = 0;
    for (int l = 0; l < p.n_layers; ++l) total += p.layer[l].do_bias ? (p.layer[l].z_on_m ? p.layer[l].d_m : p.layer[l].d_n) : 0;
    for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < total; w += (gridDim.x * blockDim.x) >> 5) {
        int l = 0, o = w;
        for (; l < p.n_layers; ++l) {
            const int n = p.layer[l].do_bias ? (p.layer[l].z_on_m ? p.layer[l].d_m : p.layer[l].d_n) : 0;
            if (o < n) break;
            o -= n;
        }
        const Layer& y = p.layer[l];
        const int width = y.z_on_m ? BM : y.N, zt = o / width, col = o - zt * width;
        const int others = y.z_on_m ? y.tiles_n : y.tiles_m;
        float acc = 0.f;
        for (int x = lane; x < others; x += 32) {
            const int t = (y.z_on_m ? zt * y.tiles_n + x : x * y.tiles_n + zt) - y.tile0;
            if (t < 0 || t >= y.tiles) continue;
            const int u0 = y.unit_base + t * y.nkb;
            const int r0 = run_of(u0), r1 = run_of(u0 + y.nkb - 1);
            for (int r = r0; r <= r1; ++r) acc += p.bias_part[(size_t)(y.tile_base + t + r) * 256 + col];
        }
        acc = warp_sum(acc);
        if (lane != 0) continue;
        if (!p.first_chunk) acc += y.gb[o];
        if (p.last_chunk && p.noise_scale > 0.f) {
            float z[4];
            normals_at((size_t)(o & ~3), y.sb0, y.sb1, p.k0, p.k1, z);
            acc = fmaf(p.noise_scale, z[o & 3], acc);
        }
        y.gb[o] = acc;
    }
}

}  // namespace tc
}  // namespace dpclip
