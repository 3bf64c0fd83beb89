// C ABI of libdpclip: argument checking, method selection and kernel launches.
#include <stdint.h>
#include <string.h>

#include "common.cuh"
#include <math.h>

#include "kernels_simt.cuh"
#include "kernels_stream.cuh"
#include "kernels_tc.cuh"
#include "kernels_tc_pair.cuh"
#include "kernels_fused_t1_tf32.cuh"
#include "kernels_tf32.cuh"
#include "kernels_group.cuh"
#include "kernels_t1_planes.cuh"
#include "kernels_fused_t1.cuh"
#include "kernels_narrow.cuh"
#include "kernels_narrow_tc.cuh"
#include "kernels_conv_tc.cuh"
#include "kernels_narrow_pack.cuh"
#include "kernels_elementwise.cuh"
#include "kernels_stage.cuh"
#include "kernels_t1_thin.cuh"

#include <stdio.h>
#include <stdlib.h>
#include <atomic>

using namespace dpclip;

namespace {

inline size_t elt_size(dpclip_dtype dt) { return dt == DPCLIP_F32 ? 4 : 2; }
inline bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
// Kernels launched by this library since it was loaded (observability only; never read by a kernel).
std::atomic<unsigned long long> g_launches{0};
constexpr int kGridCounterOffset = 64;   // workspace header: status word at 0, grid-barrier counter here
constexpr int kWorkCounterOffset = 128;  // item counter of the dynamically scheduled Gram kernel (wraps to zero by itself)
constexpr int kTailCounterOffset = 192;  // CTAs done, for the factors tail of a Gram launch (reset by the last CTA)
inline int launch_status() {
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? DPCLIP_OK : DPCLIP_ERR_CUDA;
}

// Path switches for tests and measurements (not configuration): a bit mask read ONCE from the DPCLIP_*
// environment variables, on the first call that asks, so that no entry point touches the environment on its
// way to a launch.  dpclip_reload_path_switches() re-reads them (the tests flip a variable, reload, and
// reload again afterwards).
enum PathSwitch : unsigned {
    SW_FORCE_SIMT = 1u << 0, SW_NO_NARROW = 1u << 1, SW_NO_NARROW_RING = 1u << 2, SW_NO_NARROW_TC = 1u << 3,
    SW_NO_NARROW_PACK = 1u << 4, SW_NARROW_PACK_BF16 = 1u << 5, SW_NO_GRAM_Q2 = 1u << 6, SW_NO_T1_TF32 = 1u << 7,
    SW_NO_FUSED_T1 = 1u << 8, SW_NO_GRAM_GROUP = 1u << 9, SW_NO_GRAD_GROUP = 1u << 10, SW_NO_CONV_TC = 1u << 11,
    SW_NO_CONV_PATCHES = 1u << 12, SW_TILE_M1 = 1u << 13, SW_TILE_M2 = 1u << 14, SW_T1_TWO_LAUNCHES = 1u << 15, SW_NO_PAIR = 1u << 16, SW_LOG = 1u << 17, SW_NO_FACTORS_TAIL = 1u << 18, SW_NO_SM_BUDGET = 1u << 19, SW_NO_OVERLAP = 1u << 20, SW_NO_STAGE = 1u << 21, SW_NO_GRAM_PER_EX = 1u << 22, SW_NO_PAIR_JOIN = 1u << 23, SW_NO_T1_PLANES = 1u << 24,
    SW_LOADED = 1u << 31
};
std::atomic<unsigned> g_path_switches{0};
unsigned read_path_switches() {
    static const struct { const char* name; unsigned bit; char on; } table[] = {
        {"DPCLIP_FORCE_SIMT", SW_FORCE_SIMT, '1'}, {"DPCLIP_NO_NARROW", SW_NO_NARROW, '1'},
        {"DPCLIP_NO_NARROW_RING", SW_NO_NARROW_RING, '1'}, {"DPCLIP_NO_NARROW_TC", SW_NO_NARROW_TC, '1'},
        {"DPCLIP_NO_NARROW_PACK", SW_NO_NARROW_PACK, '1'}, {"DPCLIP_NARROW_PACK_BF16", SW_NARROW_PACK_BF16, '1'},
        {"DPCLIP_NO_GRAM_Q2", SW_NO_GRAM_Q2, '1'}, {"DPCLIP_NO_T1_TF32", SW_NO_T1_TF32, '1'},
        {"DPCLIP_NO_FUSED_T1", SW_NO_FUSED_T1, '1'}, {"DPCLIP_NO_GRAM_GROUP", SW_NO_GRAM_GROUP, '1'},
        {"DPCLIP_NO_GRAD_GROUP", SW_NO_GRAD_GROUP, '1'}, {"DPCLIP_NO_CONV_TC", SW_NO_CONV_TC, '1'},
        {"DPCLIP_NO_CONV_PATCHES", SW_NO_CONV_PATCHES, '1'}, {"DPCLIP_TILE_M", SW_TILE_M1, '1'},
        {"DPCLIP_TILE_M", SW_TILE_M2, '2'}, {"DPCLIP_T1_ONE_LAUNCH", SW_T1_TWO_LAUNCHES, '0'},
        {"DPCLIP_NO_PAIR", SW_NO_PAIR, '1'}, {"DPCLIP_LOG", SW_LOG, '1'},
        {"DPCLIP_NO_FACTORS_TAIL", SW_NO_FACTORS_TAIL, '1'}, {"DPCLIP_NO_SM_BUDGET", SW_NO_SM_BUDGET, '1'},
        {"DPCLIP_NO_OVERLAP", SW_NO_OVERLAP, '1'}, {"DPCLIP_NO_STAGE", SW_NO_STAGE, '1'},
        {"DPCLIP_NO_GRAM_PER_EX", SW_NO_GRAM_PER_EX, '1'}, {"DPCLIP_NO_PAIR_JOIN", SW_NO_PAIR_JOIN, '1'}, {"DPCLIP_NO_T1_PLANES", SW_NO_T1_PLANES, '1'},
    };
    unsigned v = SW_LOADED;
    for (const auto& e : table) {
        const char* env = getenv(e.name);
        if (env && env[0] == e.on) v |= e.bit;
    }
    g_path_switches.store(v, std::memory_order_relaxed);
    return v;
}
inline bool path_switch(unsigned bit) {
    unsigned v = g_path_switches.load(std::memory_order_relaxed);
    if (!(v & SW_LOADED)) v = read_path_switches();
    return (v & bit) != 0;
}

// SM budget of the calling thread's next launches (0 = the whole GPU).  A step that spreads small layers over
// several streams gives each launch a share of the SMs in proportion to its bytes: launches of a few
// megabytes are chains of round trips, not throughput problems, so running four of them side by side on a
// quarter of the SMs each costs each one little and hides the others' latency; launched at full width they
// queue for the SMs (one CTA per SM) and run one after the other.
thread_local int t_sm_budget = 0;
inline int sm_budget() { return t_sm_budget > 0 && t_sm_budget < kNumSMs ? t_sm_budget : kNumSMs; }
// Set while the next clipped-sum launch of this thread directly follows, in its stream, the Gram launch whose tail
// computed the factors: the launch then asks for programmatic serialization (see griddep_wait in tc_common.cuh).
thread_local bool t_overlap_prev = false;
struct OverlapPrevScope {
    bool prev;
    explicit OverlapPrevScope(bool on) : prev(t_overlap_prev) { t_overlap_prev = on; }
    ~OverlapPrevScope() { t_overlap_prev = prev; }
};
struct SmBudgetScope {
    int prev;
    explicit SmBudgetScope(int b) : prev(t_sm_budget) { t_sm_budget = b; }
    ~SmBudgetScope() { t_sm_budget = prev; }
};

// Set while a step runs its norm stage with all rows of sq already at zero: launches that add their norms up with atomics then
// leave out their own clear.
thread_local bool t_sq_cleared = false;
struct SqClearedScope {
    bool prev;
    explicit SqClearedScope(bool on) : prev(t_sq_cleared) { t_sq_cleared = on; }
    ~SqClearedScope() { t_sq_cleared = prev; }
};
inline bool clear_sq(float* sq, size_t n, cudaStream_t st) {
    return t_sq_cleared || cudaMemsetAsync(sq, 0, sizeof(float) * n, st) == cudaSuccess;
}

// Launch with programmatic serialization: for kernels that call griddep_wait, right behind another kernel of their stream.
template <typename... P, typename... A>
inline int launch_behind(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, const A&... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = dim3(block); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = path_switch(SW_NO_OVERLAP) ? 0 : 1;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) { cudaGetLastError(); return DPCLIP_ERR_CUDA; }
    return launch_status();
}
// Dynamic shared memory that lets no more CTAs of a launch stand on one SM than its share of them.  Placed while the kernel in front
// leaves the SMs one after the other, a launch of few CTAs would be packed on the first.
inline int spread_smem(long blocks, int static_bytes) {
    const long k = ceil_div(blocks, (long)kNumSMs);
    return (int)((228 * 1024 / k - 1024 - static_bytes) / 1024 * 1024);
}
// The kernel that this thread is about to launch directly follows one of the same step in its stream (takes the flag).
inline bool take_overlap() { const bool on = t_overlap_prev; t_overlap_prev = false; return on; }

// DPCLIP_LOG=1: one line on stderr per dispatch decision (which form of a kernel a layer takes and how its
// work is cut) -- host side only, nothing changes on the device.
#define DPCLIP_LOGF(...) do { if (path_switch(SW_LOG)) { fprintf(stderr, "[dpclip] " __VA_ARGS__); fputc('\n', stderr); } } while (0)

int check_layer_args(const void* A, long lda, const void* Z, long ldz, int B, int T, int d_in, int d_out,
                     dpclip_dtype dtype) {
    if (!A || !Z) return DPCLIP_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || d_in <= 0 || d_out <= 0) return DPCLIP_ERR_INVALID_ARG;
    if (lda < d_in || ldz < d_out) return DPCLIP_ERR_INVALID_ARG;
    if (dtype != DPCLIP_F32 && dtype != DPCLIP_BF16) return DPCLIP_ERR_INVALID_ARG;
    if ((long)B * T > 0x7FFFFFFFL) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(A, elt_size(dtype)) || !aligned_to(Z, elt_size(dtype))) return DPCLIP_ERR_MISALIGNED;
    return DPCLIP_OK;
}

// 4-element vector loads need the base and every row start on a 4-element boundary.
inline int vec4_ok(const void* p, long ld, dpclip_dtype dt) {
    return aligned_to(p, 4 * elt_size(dt)) && (ld % 4 == 0);
}

void fill_simt_params(SimtParams& p, const void* A, long lda, const void* Z, long ldz, int T, int d_in,
                      int d_out, int has_bias, dpclip_dtype dtype) {
    memset(&p, 0, sizeof(p));
    p.A = A; p.lda = lda; p.Z = Z; p.ldz = ldz;
    p.T = T; p.d_in = d_in; p.d_out = d_out; p.has_bias = has_bias ? 1 : 0;
    p.tiles_m = ceil_div(d_out, SIMT_BM);
    p.tiles_n = ceil_div(d_in + p.has_bias, SIMT_BN);
    p.vec_a = vec4_ok(A, lda, dtype);
    p.vec_z = vec4_ok(Z, ldz, dtype);
}

int launch_t1_norms(const void* A, long lda, const void* Z, long ldz, int B, int d_in, int d_out,
                    dpclip_dtype dtype, int has_bias, float* sq, cudaStream_t st) {
    const int va = vec4_ok(A, lda, dtype), vz = vec4_ok(Z, ldz, dtype);
    if (dtype == DPCLIP_F32)
        t1_sqnorm_kernel<float><<<B, 256, 0, st>>>((const float*)A, lda, (const float*)Z, ldz, d_in, d_out,
                                                   has_bias, va, vz, sq);
    else
        t1_sqnorm_kernel<__nv_bfloat16><<<B, 256, 0, st>>>((const __nv_bfloat16*)A, lda,
                                                           (const __nv_bfloat16*)Z, ldz, d_in, d_out,
                                                           has_bias, va, vz, sq);
    return launch_status();
}

// narrow layers (d_in + bias <= 32, d_out <= 64, T > 1): streaming kernel with one lane per column
inline bool narrow_layer(int T, int d_in, int d_out, int has_bias, long lda, long ldz) {
    if (path_switch(SW_NO_NARROW)) return false;
    // dense rows: a run of rows is then one contiguous run of memory, which is what the kernel streams
    return T > 1 && d_in + (has_bias ? 1 : 0) <= 32 && d_out <= 64 && lda == d_in && ldz == d_out;
}

template <typename T, int MAXM, bool GRAD>
int launch_narrow_inst(const NarrowParams& p, int grid, cudaStream_t st) {
    constexpr int smem = NarrowCfg<MAXM>::SMEM_BYTES;
    if (cudaFuncSetAttribute(narrow_kernel<T, MAXM, GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
        cudaSuccess) return DPCLIP_ERR_CUDA;
    narrow_kernel<T, MAXM, GRAD><<<grid, NARROW_THREADS, smem, st>>>(p);
    return launch_status();
}

template <int MAXM, int WARPS, bool GRAD>
int launch_narrow_ring_inst(const NarrowParams& p, int grid, cudaStream_t st) {
    constexpr int smem = NarrowRingCfg<MAXM, WARPS>::SMEM_BYTES;
    if (cudaFuncSetAttribute(narrow_ring_kernel<MAXM, WARPS, GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
        cudaSuccess) return DPCLIP_ERR_CUDA;
    narrow_ring_kernel<MAXM, WARPS, GRAD><<<grid, 32 * WARPS, smem, st>>>(p);
    return launch_status();
}

// fp32 with every 16-row chunk starting on a 16-byte boundary (in A and in Zb): the cp.async ring form
inline bool narrow_ring_ok(const NarrowParams& p, dpclip_dtype dtype, bool grad) {
    if (path_switch(SW_NO_NARROW_RING)) return false;
    if (dtype != DPCLIP_F32 || !aligned_to(p.A, 16) || !aligned_to(p.Z, 16)) return false;
    // chunk starts are multiples of 16 rows from the slice start: 16 * d * 4 bytes is always a multiple of 16;
    // the slice start itself is a multiple of 32 rows (GRAD) or of T rows (NORM)
    if (!grad && (((long)p.T * p.d_in) % 4 != 0 || ((long)p.T * p.d_out) % 4 != 0)) return false;
    return true;
}

// bf16 narrow layers on the tensor cores: needs the status word of a workspace for its bounded waits, and
// items (examples, row slices) that start and end on 16-byte boundaries in both inputs, which the bulk copies
// into shared memory ask for
inline bool narrow_tc_ok(const NarrowParams& p, dpclip_dtype dtype, const int* status) {
    if (path_switch(SW_NO_NARROW_TC)) return false;
    if (dtype != DPCLIP_BF16 || status == nullptr) return false;
    if (!aligned_to(p.A, 16) || !aligned_to(p.Z, 16)) return false;
    return ((long)p.T * p.d_in) % 8 == 0 && ((long)p.T * p.d_out) % 8 == 0;
}

template <bool GRAD>
int launch_narrow_tc(const NarrowParams& p, int grid, int n_items, int* status, cudaStream_t st) {
    namespace n = tc::ntc;
    n::Params q;
    memset(&q, 0, sizeof(q));
    q.A = static_cast<const __nv_bfloat16*>(p.A); q.Z = static_cast<const __nv_bfloat16*>(p.Z);
    q.T = p.T; q.d_in = p.d_in; q.d_out = p.d_out; q.has_bias = p.has_bias;
    q.n_items = n_items; q.rows_total = p.rows_total; q.rows_per_cta = p.rows_per_cta;
    q.clip = p.clip; q.sq = p.sq; q.part = p.part; q.part_m = p.d_out <= 32 ? 32 : 64;
    q.status = status;
    if (!GRAD && p.d_out > 32 && !clear_sq(p.sq, (size_t)n_items, st))
        return DPCLIP_ERR_CUDA;
    if (cudaFuncSetAttribute(tc::narrow_tc_kernel<GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, n::SMEM_BYTES) !=
        cudaSuccess) return DPCLIP_ERR_CUDA;
    tc::narrow_tc_kernel<GRAD><<<grid, n::THREADS, n::SMEM_BYTES, st>>>(q);
    return launch_status();
}

// Narrow layers with d_out <= 32 on the tensor cores, four row groups per instruction (either dtype): the same
// conditions as narrow_tc_ok, on 16-byte multiples of the element size
inline bool narrow_pack_ok(const NarrowParams& p, dpclip_dtype dtype, const int* status) {
    if (path_switch(SW_NO_NARROW_TC)) return false;
    if (path_switch(SW_NO_NARROW_PACK)) return false;
    if (status == nullptr || p.d_out > 32 || p.d_in + p.has_bias > 32) return false;
    if (dtype == DPCLIP_BF16) {
        // bf16 has few instructions to save (one per 16 rows) and pays for the extra pass through shared memory in
        // the epilogue: measured 16.4 / 18.0 us against 15.2 / 17.9 us for the unpacked kernel on the first
        // convolution of the CNN.  Kept selectable for measurements.
        if (!path_switch(SW_NARROW_PACK_BF16)) return false;
    }
    if (!aligned_to(p.A, 16) || !aligned_to(p.Z, 16)) return false;
    const long es = elt_size(dtype);
    return ((long)p.T * p.d_in * es) % 16 == 0 && ((long)p.T * p.d_out * es) % 16 == 0;
}

template <typename T, bool GRAD>
int launch_narrow_pack_inst(const tc::npk::Params& q, int grid, cudaStream_t st) {
    using Cfg = tc::npk::Cfg<T>;
    if (cudaFuncSetAttribute(tc::narrow_pack_kernel<T, GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             Cfg::SMEM_BYTES) != cudaSuccess) return DPCLIP_ERR_CUDA;
    tc::narrow_pack_kernel<T, GRAD><<<grid, tc::npk::THREADS, Cfg::SMEM_BYTES, st>>>(q);
    return launch_status();
}

template <bool GRAD>
int launch_narrow_pack(const NarrowParams& p, int grid, int n_items, dpclip_dtype dtype, int* status, cudaStream_t st) {
    tc::npk::Params q;
    memset(&q, 0, sizeof(q));
    q.A = p.A; q.Z = p.Z; q.T = p.T; q.d_in = p.d_in; q.d_out = p.d_out; q.has_bias = p.has_bias;
    q.n_items = n_items; q.rows_total = p.rows_total; q.rows_per_cta = p.rows_per_cta;
    q.clip = p.clip; q.sq = p.sq; q.part = p.part; q.status = status;
    if (!GRAD && !clear_sq(p.sq, (size_t)n_items, st)) return DPCLIP_ERR_CUDA;
    return dtype == DPCLIP_F32 ? launch_narrow_pack_inst<float, GRAD>(q, grid, st)
                               : launch_narrow_pack_inst<__nv_bfloat16, GRAD>(q, grid, st);
}

template <bool GRAD>
int launch_narrow(const NarrowParams& p, int grid, int d_out, dpclip_dtype dtype, cudaStream_t st) {
    if (narrow_ring_ok(p, dtype, GRAD)) {
        // two 8-warp CTAs per SM when there are CTAs enough for that, else one 16-warp CTA
        if (grid > kNumSMs)
            return d_out <= 32 ? launch_narrow_ring_inst<32, 8, GRAD>(p, grid, st) : launch_narrow_ring_inst<64, 8, GRAD>(p, grid, st);
        return d_out <= 32 ? launch_narrow_ring_inst<32, 16, GRAD>(p, grid, st) : launch_narrow_ring_inst<64, 16, GRAD>(p, grid, st);
    }
    if (dtype == DPCLIP_F32)
        return d_out <= 32 ? launch_narrow_inst<float, 32, GRAD>(p, grid, st) : launch_narrow_inst<float, 64, GRAD>(p, grid, st);
    return d_out <= 32 ? launch_narrow_inst<__nv_bfloat16, 32, GRAD>(p, grid, st)
                       : launch_narrow_inst<__nv_bfloat16, 64, GRAD>(p, grid, st);
}

int launch_simt_norms(const void* A, long lda, const void* Z, long ldz, int B, int T, int d_in, int d_out,
                      dpclip_dtype dtype, int has_bias, float* sq, cudaStream_t st, int* status = nullptr) {
    if (narrow_layer(T, d_in, d_out, has_bias, lda, ldz)) {
        NarrowParams q;
        memset(&q, 0, sizeof(q));
        q.A = A; q.lda = lda; q.Z = Z; q.ldz = ldz; q.T = T; q.d_in = d_in; q.d_out = d_out;
        q.has_bias = has_bias ? 1 : 0; q.sq = sq;
        if (narrow_pack_ok(q, dtype, status))
            return launch_narrow_pack<false>(q, B < sm_budget() ? B : sm_budget(), B, dtype, status, st);
        if (narrow_tc_ok(q, dtype, status))
            return launch_narrow_tc<false>(q, B < sm_budget() ? B : sm_budget(), B, status, st);
        return launch_narrow<false>(q, B, d_out, dtype, st);
    }
    SimtParams p;
    fill_simt_params(p, A, lda, Z, ldz, T, d_in, d_out, has_bias, dtype);
    const int n_tiles = p.tiles_m * p.tiles_n;
    int split = ceil_div(2 * kNumSMs, B);
    if (split > n_tiles) split = n_tiles;
    if (split < 1) split = 1;
    p.sq = sq;
    p.use_atomic = split > 1;
    if (p.use_atomic && !clear_sq(sq, (size_t)B, st))
        return DPCLIP_ERR_CUDA;
    dim3 grid(split, B);
    if (dtype == DPCLIP_F32) zta_simt_kernel<float, false><<<grid, SIMT_THREADS, 0, st>>>(p);
    else zta_simt_kernel<__nv_bfloat16, false><<<grid, SIMT_THREADS, 0, st>>>(p);
    return launch_status();
}

// after_sum: the result has to be that of the sum followed by the noise, bit for bit
struct NoiseSpec { float scale; unsigned long long seed, sid_w, sid_b; bool after_sum = false; };

// noise in the epilogue of the fp32-ALU kernel; it indexes the dense tensor
void simt_noise(SimtParams& p, const NoiseSpec* noise, bool* noise_done) {
    if (!noise || !(noise->scale > 0.f) || p.ldg != p.d_in) return;
    p.noise_scale = noise->scale;
    p.k0 = (uint32_t)noise->seed; p.k1 = (uint32_t)(noise->seed >> 32);
    p.sw0 = (uint32_t)noise->sid_w; p.sw1 = (uint32_t)(noise->sid_w >> 32);
    p.sb0 = (uint32_t)noise->sid_b; p.sb1 = (uint32_t)(noise->sid_b >> 32);
    if (noise_done) *noise_done = true;
}

// T = 1 layers of at most 16 outputs (kernels_t1_thin.cuh) while a warp's rows are few, or where the tile kernel has as many tiles
// as there are SMs and gains nothing from its slices of rows.  Call with noise, thin / tile kernel, 10 outputs: bf16, 1024 inputs, B =
// 192: 12.3 / 16.3 us, 256: 15.4 / 16.4 (301 inputs, element by element: 17.8 / 16.8), 320: 19.0 / 16.6, 1024: 56 / 18; 4096 inputs, 1024: 56 / 31,
// 16384: 59 / 97.  fp32, 1024 inputs, 320: 12.7 / 15.4, 384: 14.7 / 15.4 (301 inputs: 16.4 / 15.7), 512: 18.9 / 15.4; 4096 inputs, 512: 18.8 / 27.7,
// 1024: 35.7 / 37.6.
inline bool t1_thin_pairs(const void* A, long lda, dpclip_dtype dtype) { return aligned_to(A, 2 * elt_size(dtype)) && lda % 2 == 0; }
inline bool t1_thin_ok(const void* A, long lda, int B, int T, int d_in, int d_out, dpclip_dtype dtype) {
    if (T != 1 || d_out > THIN_OUT || B > 1024 || path_switch(SW_FORCE_SIMT)) return false;
    const bool pairs = t1_thin_pairs(A, lda, dtype);
    return dtype == DPCLIP_F32 ? B <= (pairs ? 384 : 360) || d_in >= 4096 : B <= (pairs ? 256 : 240) || d_in >= 9216;
}
int launch_t1_thin_grad(const void* A, long lda, const void* Z, long ldz, int B, int d_in, int d_out, dpclip_dtype dtype,
                        const float* clip, float* gW, long ldg, float* gb, cudaStream_t st, const NoiseSpec* noise, bool* noise_done) {
    ThinParams p;
    memset(&p, 0, sizeof(p));
    p.A = A; p.lda = lda; p.Z = Z; p.ldz = ldz; p.B = B; p.d_in = d_in; p.d_out = d_out;
    p.pairs_ok = t1_thin_pairs(A, lda, dtype);
    p.clip = clip; p.gW = gW; p.ldg = ldg; p.gb = gb;
    if (noise && noise->scale > 0.f && ldg == d_in) {
        p.noise_scale = noise->scale;
        p.k0 = (uint32_t)noise->seed; p.k1 = (uint32_t)(noise->seed >> 32);
        p.sw0 = (uint32_t)noise->sid_w; p.sw1 = (uint32_t)(noise->sid_w >> 32);
        p.sb0 = (uint32_t)noise->sid_b; p.sb1 = (uint32_t)(noise->sid_b >> 32);
        if (noise_done) *noise_done = true;
    }
    const int grid = ceil_div(d_in, (long)THIN_COLS);
    if (dtype == DPCLIP_F32) t1_thin_grad_kernel<float><<<grid, THIN_THREADS, 0, st>>>(p);
    else t1_thin_grad_kernel<__nv_bfloat16><<<grid, THIN_THREADS, 0, st>>>(p);
    return launch_status();
}

int launch_simt_grad(const void* A, long lda, const void* Z, long ldz, int B, int T, int d_in, int d_out,
                     dpclip_dtype dtype, const float* clip, float* gW, long ldg, float* gb, cudaStream_t st,
                     void* workspace = nullptr, size_t workspace_bytes = 0, const NoiseSpec* noise = nullptr,
                     bool* noise_done = nullptr) {
    if (narrow_layer(T, d_in, d_out, gb != nullptr, lda, ldz)) {
        NarrowParams q;
        memset(&q, 0, sizeof(q));
        q.A = A; q.lda = lda; q.Z = Z; q.ldz = ldz; q.T = T; q.d_in = d_in; q.d_out = d_out;
        q.has_bias = gb ? 1 : 0; q.clip = clip; q.gW = gW; q.ldg = ldg; q.gb = gb;
        q.rows_total = (long)B * T;
        int* status = (workspace && workspace_bytes >= (size_t)kHeaderBytes) ? static_cast<int*>(workspace) : nullptr;
        const bool on_pack = narrow_pack_ok(q, dtype, status);
        const bool on_tc = on_pack || narrow_tc_ok(q, dtype, status);
        // one wave: a CTA of the register-staged kernel holds a whole SM; the cp.async form runs two per SM
        int grid = (!on_tc && narrow_ring_ok(q, dtype, true)) ? 2 * sm_budget() : sm_budget();
        const long min_rows = NARROW_WARPS * 32;                   // at least one chunk per warp
        if ((long)grid * min_rows > q.rows_total) grid = (int)((q.rows_total + min_rows - 1) / min_rows);
        // whole 32-row chunks per CTA: every chunk of a dense layer then starts on a 16-byte boundary whatever
        // the row length, and takes the 128-bit load path (a slice starting mid-chunk falls back to scalar loads)
        q.rows_per_cta = ((q.rows_total + grid - 1) / grid + 31) / 32 * 32;
        grid = (int)((q.rows_total + q.rows_per_cta - 1) / q.rows_per_cta);
        const int maxm = d_out <= 32 ? 32 : 64;
        const int parts_per_cta = 1;
        const size_t part_bytes = (size_t)grid * parts_per_cta * maxm * 32 * 4;
        if (workspace && workspace_bytes >= (size_t)kHeaderBytes + part_bytes && grid > 1) {
            // partial tile per CTA, then a fixed-order reduce that also adds the noise
            q.part = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes);
            int rc = on_pack ? launch_narrow_pack<true>(q, grid, 1, dtype, status, st)
                   : on_tc   ? launch_narrow_tc<true>(q, grid, 1, status, st)
                             : launch_narrow<true>(q, grid, d_out, dtype, st);
            if (rc) return rc;
            NarrowReduceParams r;
            memset(&r, 0, sizeof(r));
            r.part = q.part; r.n_parts = grid * parts_per_cta; r.maxm = maxm; r.d_out = d_out; r.d_in = d_in; r.has_bias = gb ? 1 : 0;
            r.gW = gW; r.ldg = ldg; r.gb = gb;
            if (noise && noise->scale > 0.f && ldg == d_in) {
                r.noise_scale = noise->scale;
                r.k0 = (uint32_t)noise->seed; r.k1 = (uint32_t)(noise->seed >> 32);
                r.sid_w = noise->sid_w; r.sid_b = noise->sid_b;
                if (noise_done) *noise_done = true;
            }
            return launch_behind(narrow_reduce_kernel, dim3(d_out), 256, 0, st, r);
        }
        if (cudaMemset2DAsync(gW, sizeof(float) * (size_t)ldg, 0, sizeof(float) * (size_t)d_in, d_out, st) !=
            cudaSuccess) return DPCLIP_ERR_CUDA;
        if (gb && cudaMemsetAsync(gb, 0, sizeof(float) * (size_t)d_out, st) != cudaSuccess) return DPCLIP_ERR_CUDA;
        return launch_narrow<true>(q, grid, d_out, dtype, st);
    }
    if (t1_thin_ok(A, lda, B, T, d_in, d_out, dtype))
        return launch_t1_thin_grad(A, lda, Z, ldz, B, d_in, d_out, dtype, clip, gW, ldg, gb, st, noise, noise_done);
    SimtParams p;
    fill_simt_params(p, A, lda, Z, ldz, T, d_in, d_out, gb != nullptr, dtype);
    const int n_tiles = p.tiles_m * p.tiles_n;
    const long rows = (long)B * T;
    long ksplit = ceil_div(4 * kNumSMs, n_tiles);
    const long max_split = (rows + 4 * SIMT_BK - 1) / (4 * SIMT_BK);     // at least 64 rows per slice
    if (ksplit > max_split) ksplit = max_split;
    if (ksplit < 1) ksplit = 1;
    if (ksplit > 65535) ksplit = 65535;
    long per = (rows + ksplit - 1) / ksplit;
    per = (per + SIMT_BK - 1) / SIMT_BK * SIMT_BK;
    ksplit = (rows + per - 1) / per;
    p.clip = clip; p.gW = gW; p.ldg = ldg; p.gb = gb;
    p.rows_total = rows; p.rows_per_split = per;
    p.use_atomic = ksplit > 1;
    if (p.use_atomic) {
        if (cudaMemset2DAsync(gW, sizeof(float) * (size_t)ldg, 0, sizeof(float) * (size_t)d_in, d_out, st) !=
            cudaSuccess) return DPCLIP_ERR_CUDA;
        if (gb && cudaMemsetAsync(gb, 0, sizeof(float) * (size_t)d_out, st) != cudaSuccess)
            return DPCLIP_ERR_CUDA;
    }
    // slices add up in any order, the noise among them
    if (ksplit == 1 || !noise || !noise->after_sum) simt_noise(p, noise, noise_done);
    dim3 grid(n_tiles, (unsigned)ksplit);
    if (dtype == DPCLIP_F32) zta_simt_kernel<float, true><<<grid, SIMT_THREADS, 0, st>>>(p);
    else zta_simt_kernel<__nv_bfloat16, true><<<grid, SIMT_THREADS, 0, st>>>(p);
    return launch_status();
}


// ---------------------------------------------------------------------------
// tensor-core paths (bf16): tensor maps + launches
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;       // a driver entry point, looked up once; not device state
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// 2-D bf16 matrix [rows][cols] with row stride ld elements; box = box_cols x box_rows, 128-byte swizzle,
// out-of-range elements read as zero.
bool make_map_bf16(CUtensorMap* map, const void* base, long rows, long cols, long ld, int box_cols, int box_rows,
                   bool swizzle = true) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// TMA needs 16-byte aligned bases and row strides.
inline bool tc_eligible(const void* A, long lda, const void* Z, long ldz, dpclip_dtype dtype) {
    if (dtype != DPCLIP_BF16) return false;
    if (path_switch(SW_FORCE_SIMT)) return false;
    return aligned_to(A, 16) && aligned_to(Z, 16) && lda % 8 == 0 && ldz % 8 == 0;
}

template <typename K>
bool enable_smem(K kernel, int bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
}
// The same for a kernel whose SMs small launches on other streams may share: the smallest division of L1 and shared memory that
// holds the kernel (196 KB for a Gram kernel) would leave those none.  One transformer block (B = 128, T = 256, d = 512): the norms
// of its LayerNorms ran behind the Gram launch, 100 to 135 us; beside it they end at 111 us, the Gram launch at 129 instead of 114.
template <typename K>
bool enable_smem_shared(K kernel, int bytes) {
    return enable_smem(kernel, bytes) &&
           cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess;
}

// One layer of a Gram-norm launch.
struct GramLayer {
    const void* A; long lda; const void* Z; long ldz;
    int B, T, d_in, d_out, has_bias;
    float* sq;
    bool per_ex;                   // row blocks begin with their example (gram_per_ex)
};

// Examples of two row blocks: their own kernel, one HBM pass per example.
inline bool gram_two_blocks(int T) {
    return T == 2 * tc::gram::BM && !path_switch(SW_NO_GRAM_Q2);
}
// Row blocks that begin with their example, not with a multiple of 128 rows; width[0 .. n) are the d_in + d_out of the launch's
// layers, widest first.  Flattened over the examples, a block that crosses into the next example meets a column block more, and
// a long example was re-read from HBM; beginning with the example, its last block is partly empty and there are more work
// items.  Which takes less follows from T, B and the layers: the items are dealt to the CTAs as the launch deals them, an item
// costing one unit a feature, half a unit more for every column block and for a row block of its own, and 300 for its drain; the
// order whose busiest CTA has less to do wins, by 5 % for the re-reads of examples of several blocks, else by 2 %.
// Kernel, flattened / by example: T = 96, three layers of 1536 features, 64 examples: 17 / 24 us; T = 192, 260 examples of 1024 +
// 2560: 77 / 88; T = 200, 250: 129 / 87; T = 156, 16 of 4096: 47 / 28; T = 512, 256 of 5120: 608 / 383; T = 2048, 32 of 8192:
// 3813 / 844.  551 launches (T = 66 to 383, 16 to 320 examples, one to seven layers of 768 to 2560 features): 0.3 % over the
// faster order of each, where ranges of T alone (by example from 88 rows, but for 129 to 167 and 257 to 287) were 4.5 % over.
inline bool gram_per_ex(int T, int B, const int* width, int n) {
    namespace g = tc::gram;
    if (T <= g::BM / 2 || T == g::BM || gram_two_blocks(T) || path_switch(SW_NO_GRAM_PER_EX)) return false;
    const int q = ceil_div(T, (long)g::BM), subs = g::subs_of(q), sms = sm_budget();
    if (T >= 3 * g::BM) return (long)B * subs < 1L << 27;               // items of a launch are counted in an int
    struct Item { double features; int subs; };
    auto row_block = [](int rb, int cb_max) {                           // rb against column blocks rb .. cb_max, two at a time
        Item c = {0.0, 0};
        for (int cb = rb; cb <= cb_max; cb += 2, ++c.subs) c.features += 1.0 + (cb < cb_max ? 1.0 : 0.5) + (cb > rb ? 0.5 : 0.0);
        return c;
    };
    // steady: the period divides the number of CTAs, so a CTA always gets the same item of it
    auto busiest = [&](const Item* item, int period, long items, bool steady) {
        if (n * items <= 2400) {
            double load[kNumSMs] = {0.0}, most = 0.0;
            int cta = 0;
            for (int l = 0; l < n; ++l)
                for (long i = 0, k = 0; i < items; ++i) {
                    load[cta] += item[k].features * width[l] + 300.0 * item[k].subs;
                    if (++k == period) k = 0;
                    if (++cta == sms) cta = 0;
                }
            for (int c = 0; c < sms; ++c) most = load[c] > most ? load[c] : most;
            return most;
        }
        double mean = 0.0, most = 0.0, drains = 0.0, sum = 0.0;
        for (int k = 0; k < period; ++k) {
            mean += item[k].features / period; drains += 300.0 * item[k].subs / period;
            most = item[k].features > most ? item[k].features : most;
        }
        const double one = steady ? most : mean;
        for (int l = 0; l < n; ++l) sum += (one * width[l] + drains) * items / sms;
        const double part = (double)ceil_div(n * items, (long)sms) - (double)n * items / sms;       // of a last wave
        return sum + part * (one * width[n - 1] + drains);
    };
    Item own[4], flat[3 * g::BM];
    int k = 0;
    for (int rb = 0; rb < q; ++rb)
        for (int cb = rb; cb < q; cb += 2) own[k++] = {1.0 + (cb + 1 < q ? 1.0 : 0.5) + (cb > rb ? 0.5 : 0.0), 1};
    const long blocks = ceil_div((long)B * T, (long)g::BM);
    int period = T;                                                     // blocks after which the examples lie alike: T / gcd(T, 128)
    for (int two = 1; two < g::BM && period % 2 == 0; two *= 2) period /= 2;
    if (period > blocks) period = (int)blocks;
    for (int rb = 0, end = T - 1; rb < period; ++rb) {                  // end: last row of the block's last example
        while (end < rb * g::BM + g::BM - 1) end += T;
        flat[rb] = row_block(rb, end / g::BM);
    }
    return busiest(own, subs, (long)B * subs, true) <= busiest(flat, period, blocks, false) * (q > 1 ? 1.05 : 0.98);
}
// every item is on the diagonal when an example spans at most two aligned row blocks
inline bool gram_diag_only(int T, bool per_ex) {
    namespace g = tc::gram;
    return (per_ex && T <= 2 * g::BM) || (T % g::BM == 0 && T <= 2 * g::BM) || (g::BM % T == 0);
}

// Which Gram kernel a layer takes; layers of one class can share a launch, and the kernel of class 2 takes layers of class 1 too.
//   0: examples of exactly two row blocks (their own kernel: one HBM pass per example)
//   1: other layers whose items all sit on the diagonal (stages of two tiles, six of them)
//   2: the rest
inline int gram_class(int T, bool per_ex) {
    if (gram_two_blocks(T)) return 0;
    return gram_diag_only(T, per_ex) ? 1 : 2;
}

// Norms of up to gram::MAX_LAYERS layers by the Gram identity in ONE launch of kernel class `cls`.  Layers go in descending order of bytes per group, so that the round-robin deal
// leaves the small items for the end of every CTA's queue.
int launch_gram_group(const GramLayer* ls, int n, int cls, int* status, cudaStream_t st,
                      const tc::gram::FactorsTail* tail = nullptr) {
    namespace g = tc::gram;
    if (n <= 0 || n > g::MAX_LAYERS) return DPCLIP_ERR_INVALID_ARG;
    int order[g::MAX_LAYERS];
    for (int i = 0; i < n; ++i) order[i] = i;
    auto cost = [&](int i) { return (long)ls[i].d_in + ls[i].d_out; };
    for (int i = 1; i < n; ++i)                       // insertion sort, stable
        for (int j = i; j > 0 && cost(order[j]) > cost(order[j - 1]); --j) { const int t = order[j]; order[j] = order[j - 1]; order[j - 1] = t; }
    static_assert(sizeof(g::Launch) <= 4096, "kernel parameter space");
    g::Launch q;
    memset(&q, 0, sizeof(q));
    q.L = n; q.status = status;
    int groups = 0;
    for (int k = 0; k < n; ++k) {
        const GramLayer& y = ls[order[k]];
        const int own = gram_class(y.T, y.per_ex);
        if (own != cls && !(cls == 2 && own == 1)) return DPCLIP_ERR_INVALID_ARG;
        const long R = (long)y.B * y.T;
        if (!make_map_bf16(&q.map_a[k], y.A, R, y.d_in, y.lda, g::BK, g::BM) ||
            !make_map_bf16(&q.map_z[k], y.Z, R, y.d_out, y.ldz, g::BK, g::BM))
            return DPCLIP_ERR_CUDA;
        g::Params& p = q.layer[k];
        p.R = (int)R; p.T = y.T; p.d_in = y.d_in; p.d_out = y.d_out; p.has_bias = y.has_bias ? 1 : 0;
        p.sq = y.sq;
        if (cls == 0) {
            p.n_groups = y.B;                     // one example per group
        } else if (y.per_ex) {
            p.per_ex = 1; p.q = ceil_div(y.T, g::BM); p.subs = g::subs_of(p.q);
            p.n_groups = y.B * p.subs;
        } else {
            p.n_groups = ceil_div(R, g::BM);      // one 128-row block per group
        }
        q.group_begin[k] = groups;
        groups += p.n_groups;
    }
    // the general kernels accumulate with atomics: clear the rows, adjacent rows of sq in one memset (the kernel
    // for examples of two row blocks stores every norm, so its rows need no clearing)
    if (cls != 0) {
        int by_ptr[g::MAX_LAYERS];
        for (int i = 0; i < n; ++i) by_ptr[i] = i;
        for (int i = 1; i < n; ++i)
            for (int j = i; j > 0 && ls[by_ptr[j]].sq < ls[by_ptr[j - 1]].sq; --j) { const int t = by_ptr[j]; by_ptr[j] = by_ptr[j - 1]; by_ptr[j - 1] = t; }
        for (int i = 0; i < n;) {
            float* begin = ls[by_ptr[i]].sq;
            float* end = begin + ls[by_ptr[i]].B;
            int j = i + 1;
            while (j < n && ls[by_ptr[j]].sq == end) { end += ls[by_ptr[j]].B; ++j; }
            if (!clear_sq(begin, (size_t)(end - begin), st)) return DPCLIP_ERR_CUDA;
            i = j;
        }
    }
    q.group_begin[n] = groups;
    q.total_groups = groups;
    if (tail) {
        q.tail = *tail;
        q.tail.done = reinterpret_cast<unsigned int*>(reinterpret_cast<char*>(status) + kTailCounterOffset);
    }
    const int grid = groups < sm_budget() ? groups : sm_budget();
    if (cls == 0) q.work_counter = reinterpret_cast<unsigned int*>(reinterpret_cast<char*>(status) + kWorkCounterOffset);
    const auto kernel = cls == 0 ? tc::gram_norm_q2_kernel : cls == 1 ? tc::gram_norm_kernel<true> : tc::gram_norm_kernel<false>;
    if (!enable_smem_shared(kernel, g::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
    if (take_overlap()) return launch_behind(kernel, dim3(grid), g::THREADS, g::SMEM_BYTES, st, q);
    kernel<<<grid, g::THREADS, g::SMEM_BYTES, st>>>(q);
    return launch_status();
}

int launch_gram_norms(const void* A, long lda, const void* Z, long ldz, int B, int T, int d_in, int d_out,
                      int has_bias, float* sq, int* status, cudaStream_t st) {
    const int width = d_in + d_out;
    const bool per_ex = gram_per_ex(T, B, &width, 1);
    const GramLayer y = {A, lda, Z, ldz, B, T, d_in, d_out, has_bias, sq, per_ex};
    return launch_gram_group(&y, 1, gram_class(T, per_ex), status, st);
}

// Largest scratch the split-row clipped sum can ask for: one partial tile per item, at most one
// wave of 256 x 256 tiles or two waves of 128 x 256 tiles, plus the partial bias sums.
constexpr size_t kTcScratchBytes = (size_t)kNumSMs * 256 * 256 * 4 + (size_t)2 * kNumSMs * 256 * 4;

// Row split of the bf16 tensor-core clipped sum: how many row slices each output tile is cut into.
//   one wave  : floor(per_sm * SMs / tiles) slices -- every CTA one item (two for the small tile when they
//               stay long); its partial tiles fit the fixed scratch above.
//   preferred : when one wave would leave more than 5 % of the SMs idle (64 tiles of 256 x 256: 128 of 148)
//               and the row ranges stay long (>= 192 stages of 64 rows, so that pipeline fill and epilogue
//               stay below 4 % of an item), the smallest split whose items fill whole waves to >= 97 %; it
//               needs one partial tile per item, which the workspace query reports for the layer.
struct ZtaSplit { int one_wave, preferred; };
inline ZtaSplit zta_pick_split(long nkb, int tiles, int per_sm, int slots = kNumSMs) {
    ZtaSplit r;
    long base = ((long)per_sm * slots) / tiles;
    if (base > nkb) base = nkb;
    if (base < 1) base = 1;
    r.one_wave = r.preferred = (int)base;
    auto fill = [&](long ks) {
        const long items = (long)tiles * ks, waves = (items + slots - 1) / slots;
        return (double)items / (double)(waves * slots);
    };
    double best = fill(base);
    if (per_sm != 1 || best >= 0.95) return r;
    for (long ks = base + 1; ks <= 64 * base && nkb / ks >= 192; ++ks) {
        const double f = fill(ks);
        if (f > best + 0.01) { best = f; r.preferred = (int)ks; if (f >= 0.97) break; }
    }
    return r;
}
inline size_t zta_scratch_bytes(int tiles, int ksplit, int BM, bool bias) {
    return (size_t)tiles * ksplit * ((size_t)BM * 256 * 4 + (bias ? (size_t)BM * 4 : 0));
}

// second stage of a split-row clipped sum: fixed-order sum of the partial tiles (+ optional noise)
// Layers of one shape that share a clipped-sum launch (n == 0: a single layer).
struct GradGroup {
    int n;
    float* gW[tc::zta::MAX_LAYERS]; float* gb[tc::zta::MAX_LAYERS];
    unsigned long long sid_w[tc::zta::MAX_LAYERS], sid_b[tc::zta::MAX_LAYERS];
};

int launch_reduce_partials(const tc::zta::Params& p, int tiles, int ksplit, int BM, int BN, int d_in, int d_out,
                           float* gW, long ldg, float* gb, const NoiseSpec* noise, bool* noise_done,
                           cudaStream_t st, const GradGroup* grp = nullptr) {
    tc::ReduceParams r;
    memset(&r, 0, sizeof(r));
    if (grp && grp->n > 0) {
        r.n_layers = grp->n; r.tiles_layer = tiles / grp->n;
        for (int l = 0; l < grp->n; ++l) {
            r.gW_l[l] = grp->gW[l]; r.gb_l[l] = grp->gb[l];
            r.sw0_l[l] = (uint32_t)grp->sid_w[l]; r.sw1_l[l] = (uint32_t)(grp->sid_w[l] >> 32);
            r.sb0_l[l] = (uint32_t)grp->sid_b[l]; r.sb1_l[l] = (uint32_t)(grp->sid_b[l] >> 32);
        }
    }
    r.part = p.part; r.bias_part = p.bias_part;
    r.n_tiles = tiles; r.tiles_n = p.tiles_n; r.ksplit = ksplit; r.BM = BM; r.BN = BN;
    r.d_out = d_out; r.d_in = d_in; r.gW = gW; r.ldg = ldg; r.gb = gb; r.vec_ok = p.vec_ok;
    if (noise && noise->scale > 0.f && ldg == d_in) {
        r.noise_scale = noise->scale;
        r.k0 = (uint32_t)noise->seed; r.k1 = (uint32_t)(noise->seed >> 32);
        r.sw0 = (uint32_t)noise->sid_w; r.sw1 = (uint32_t)(noise->sid_w >> 32);
        r.sb0 = (uint32_t)noise->sid_b; r.sb1 = (uint32_t)(noise->sid_b >> 32);
        if (noise_done) *noise_done = true;
    }
    const long n_vec = (long)d_out * ((d_in + 3) / 4);
    // split the row slices over up to 8 thread rows per CTA until the grid has about two CTAs per SM
    int lanes = 1;
    while (lanes < 8 && lanes * 2 <= ksplit && n_vec * lanes < 2L * kNumSMs * 256) lanes *= 2;
    r.lanes = lanes;
    long blocks = (n_vec + (256 / lanes) - 1) / (256 / lanes);
    if (blocks > 8L * kNumSMs) blocks = 8L * kNumSMs;
    return launch_behind(tc::reduce_partials_kernel, dim3((unsigned)blocks, r.n_layers > 0 ? r.n_layers : 1), 256, 0, st, r);
}

// Tile shape: 256 x 256 (MT = 2) cuts the L2->SM traffic per flop by a third but has a single
// accumulator buffer; it pays once d_out spans at least two 128-row sub-tiles.
template <int MT, bool SPLIT = false>
int launch_zta_tc_mt(const tc::zta::Maps& maps, tc::zta::Params p, int B, bool norm_mode,
                     float* gW, long ldg, float* gb, float* sq, int d_in, int d_out, void* workspace,
                     size_t workspace_bytes, const NoiseSpec* noise, bool* noise_done, cudaStream_t st,
                     bool fit_to_workspace = false, const GradGroup* grp = nullptr) {
    namespace z = tc::zta;
    constexpr int BM = z::Cfg<MT, SPLIT>::BM;
    const long R = p.R;
    p.tiles_m_layer = ceil_div(d_out, BM);
    p.tiles_m = p.tiles_m_layer * (grp && grp->n > 0 ? grp->n : 1);
    p.tiles_n = ceil_div(d_in, z::BN);
    const int tiles = p.tiles_m * p.tiles_n;
    int ksplit = 1;
    if (norm_mode) {
        p.n_items = B * tiles;
        if (!clear_sq(sq, (size_t)B, st)) return DPCLIP_ERR_CUDA;
    } else {
        const int nkb = ceil_div(R, z::Cfg<MT>::BK);
        // One wave of equally long items: the kernel is bound by L2->SM traffic, so what matters is that
        // every SM streams the same number of row blocks.  (MT = 1 has two accumulator buffers and can
        // overlap the epilogue of one item with the next, so it takes two items per SM when they stay long.)
        const int sms = sm_budget();
        const int per_sm = (MT == 1 && tiles <= sms && nkb / ((2 * sms) / tiles) >= 16) ? 2 : 1;
        const ZtaSplit split = zta_pick_split(nkb, tiles, per_sm, sms);
        // the preferred split when the workspace holds its partial tiles, else one wave
        ksplit = split.one_wave;
        if (split.preferred != split.one_wave && !fit_to_workspace &&
            workspace_bytes >= kHeaderBytes + zta_scratch_bytes(tiles, split.preferred, BM, gb != nullptr))
            ksplit = split.preferred;
        if (fit_to_workspace) {                 // fixed-size scratch: take fewer, longer row slices
            const size_t per_item = (size_t)BM * z::BN * 4 + (gb ? (size_t)BM * 4 : 0);
            const size_t room = workspace_bytes > (size_t)kHeaderBytes ? workspace_bytes - kHeaderBytes : 0;
            const long fit = (long)(room / per_item / tiles);
            if (ksplit > fit) ksplit = (int)fit;
        }
        if (ksplit > nkb) ksplit = nkb;
        if (ksplit < 1) ksplit = 1;
        p.kb_per_split = ceil_div(nkb, ksplit);
        p.windows = ceil_div(p.kb_per_split, (long)z::SPLIT_WINDOW);
        ksplit = ceil_div(nkb, p.kb_per_split);
        p.n_items = tiles * ksplit;
        if (grp && grp->n > 0 && ksplit == 1) return 1;        // a group's outputs go through the partial tiles
        if (ksplit > 1) {
            const size_t part_bytes = (size_t)p.n_items * BM * z::BN * 4;
            const size_t bias_bytes = gb ? (size_t)p.n_items * BM * 4 : 0;
            if (workspace_bytes < kHeaderBytes + part_bytes + bias_bytes) return DPCLIP_ERR_WORKSPACE;
            p.part = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes);
            p.bias_part = gb ? p.part + part_bytes / 4 : nullptr;
        } else if (gb && cudaMemsetAsync(gb, 0, sizeof(float) * (size_t)d_out, st) != cudaSuccess) {
            return DPCLIP_ERR_CUDA;         // single item per tile: direct stores, bias by red.add
        }
    }
    if (!enable_smem(tc::zta_tc_kernel<MT, SPLIT>, z::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
    const int grid = p.n_items < sm_budget() ? p.n_items : sm_budget();
    tc::zta_tc_kernel<MT, SPLIT><<<grid, z::THREADS, z::SMEM_BYTES, st>>>(maps, p);
    int rc = launch_status();
    if (rc || norm_mode || ksplit == 1) return rc;

    return launch_reduce_partials(p, tiles, ksplit, BM, z::BN, d_in, d_out, gW, ldg, gb, noise, noise_done, st, grp);
}

// Clipped sums on CTA pairs (zta_pair_kernel): 512 x 256 tiles, the (tile, stage) units of all layers of the
// launch cut into equal runs, one per pair.  A layer qualifies when the padding of d_out to 512-row pair tiles
// costs at most a tenth more than its padding to 256-row tiles.
constexpr int kNumPairs = kNumSMs / 2;
inline bool pair_tile_ok(int d_out) {
    if (path_switch(SW_NO_PAIR) || d_out <= 256) return false;
    const double pad_pair = (double)ceil_div(d_out, 512) * 512, pad_single = (double)ceil_div(d_out, 256) * 256;
    return pad_pair <= 1.1 * pad_single;
}
inline int pair_tiles(int d_in, int d_out) { return ceil_div(d_out, tc::ztp::BM) * ceil_div(d_in, tc::ztp::BN); }
// Layers of a step that share a pair launch: besides the above, those whose padding costs a pair at most twelve stages (0.9 us
// each), because every launch of its own costs about 25 us (set-up, a short row slice per CTA, drain, reduce).  Sequence model of
// four projections d -> d, d -> f -> d and gates, in a graph, apart / shared: 2048 rows, d = 136, f = 400: 76 / 36 us (per-layer
// clipping, which had no shared launch for them: 111 / 35); 16384: 123 / 79; 32000, d = 300, f = 1100 (ten stages): 515 / 428; but
// 32000, d = 640, f = 2048 (fifteen): 557 / 572.  Not below eight stages of rows: the two kernels round a different operand to bf16
// (c a here, c zb there), and on so few rows a step's sums are held to those of the single-layer calls.
inline bool pair_shared_ok(int d_in, int d_out, long rows) {
    if (path_switch(SW_NO_PAIR)) return false;
    if (pair_tile_ok(d_out)) return true;
    const long stages = ceil_div(rows, (long)tc::ztp::BK);
    if (path_switch(SW_NO_PAIR_JOIN) || stages < 8) return false;
    const double waste = pair_tiles(d_in, d_out) - 0.25 * ceil_div(d_out, 128) * ceil_div(d_in, 256);
    return waste * stages <= 12.0 * kNumPairs;
}
inline size_t pair_segment_bytes(bool bias) {
    return tc::ztp::SEG_ELEMS * 4 + (bias ? (size_t)tc::ztp::BM * 4 : 0);
}
// scratch for a launch over `tiles` pair tiles with every pair busy: one segment per tile position of every
// super-layer (at most tiles + 15 positions when narrow layers leave a super-layer part empty) and one per pair
inline size_t pair_scratch_bytes(int tiles) { return (size_t)(tiles + 16 + kNumPairs) * pair_segment_bytes(true); }
inline long gcd_l(long a, long b) { while (b) { const long t = a % b; a = b; b = t; } return a; }

struct StreamLayer {
    const void* A; long lda; const void* Z; long ldz; int d_in, d_out;
    float* gW; long ldg; float* gb; unsigned long long sid_w, sid_b;
    const float* clip;             // this layer's factors [B], or NULL
    bool split;                    // scaled operand in two bf16 terms
};

// Returns DPCLIP_OK, a negative status, or 1 when the workspace cannot hold even one segment per tile (the
// caller then takes another path).
int launch_zta_stream(const StreamLayer* ls, int n, int B, int T, const NoiseSpec* noise,
                      bool* noise_done, void* workspace, size_t workspace_bytes, cudaStream_t st) {
    namespace zp = tc::ztp;
    if (n < 1 || n > zp::MAX_LAYERS) return 1;
    const long R = (long)B * T;
    tc::zta::Maps maps;
    zp::Params p;
    memset(&p, 0, sizeof(p));
    p.R = (int)R; p.T = T; p.S = (int)ceil_div(R, (long)zp::BK); p.n_layers = n;
    p.status = static_cast<int*>(workspace);
    bool fuse_noise = noise && noise->scale > 0.f, any_split = false, cut = false;
    int G = 0;
    for (int l = 0; l < n; ++l) {
        const StreamLayer& y = ls[l];
        if (!make_map_bf16(&maps.a[l], y.A, R, y.d_in, y.lda, 64, zp::BK) ||
            !make_map_bf16(&maps.z[l], y.Z, R, y.d_out, y.ldz, 64, zp::BK))
            return DPCLIP_ERR_CUDA;
        zp::Layer& q = p.layer[l];
        q.d_in = y.d_in; q.d_out = y.d_out;
        q.tiles_n = ceil_div(y.d_in, zp::BN);
        q.N = (int)round_up(ceil_div(y.d_in, (long)q.tiles_n), 32);
        q.tile_base = G; q.tiles = pair_tiles(y.d_in, y.d_out);
        G += q.tiles;
        q.do_bias = y.gb ? 1 : 0;
        q.clip = y.clip;
        q.split = y.split ? 1 : 0;
        any_split = any_split || y.split;
        cut = cut || q.N != zp::BN || (y.d_out - 1) % zp::BM < zp::BM_CTA;
        q.gW = y.gW; q.gb = y.gb; q.ldg = y.ldg;
        q.vec_ok = aligned_to(y.gW, 16) && y.ldg % 4 == 0;
        q.sw0 = (uint32_t)y.sid_w; q.sw1 = (uint32_t)(y.sid_w >> 32);
        q.sb0 = (uint32_t)y.sid_b; q.sb1 = (uint32_t)(y.sid_b >> 32);
        if (y.gb) p.any_bias = 1;
        // the noise of element j is indexed by its position in the dense tensor
        if (y.ldg != y.d_in) fuse_noise = false;
    }
    p.G = G;
    if (G > zp::MAX_TILES) return 1;
    // Gang width: the widest W <= 16 for which every layer either splits into whole super-layers (tiles % W == 0)
    // or is narrower than W (narrow layers are packed side by side), and whose gangs and super-layers leave at
    // most a tenth of the pairs idle; else W = 1 (tile-major, no sharing of rows between tiles).
    int W = 1, n_super = G;
    for (int w = 16; w >= 2; --w) {
        bool ok = true;
        int supers = 0, open_fill = 0;              // narrow layers: first fit into the open super-layer
        for (int l = 0; l < n && ok; ++l) {
            const int t = p.layer[l].tiles;
            if (t >= w) { ok = t % w == 0; supers += t / w; }
            else if (open_fill > 0 && open_fill + t <= w) open_fill += t;
            else { ++supers; open_fill = t; }
        }
        if (!ok || (long)supers * w > zp::MAX_TILES) continue;
        const double use = (double)(kNumPairs / w) * w / kNumPairs * ((double)G / ((double)supers * w));
        if (use >= 0.9) { W = w; n_super = supers; break; }
    }
    p.W = W; p.n_super = n_super;
    for (int i = 0; i < zp::MAX_TILES; ++i) { p.super_tile[i] = -1; p.tile_slot[i] = 0; }
    {
        int next_super = 0, open_super = -1, open_fill = 0;
        for (int l = 0; l < n; ++l) {
            const zp::Layer& q = p.layer[l];
            if (q.tiles >= W) {
                for (int t = 0; t < q.tiles; ++t) {
                    const int sl = next_super + t / W, j = t % W;
                    p.super_tile[sl * W + j] = (short)(q.tile_base + t);
                    p.tile_slot[q.tile_base + t] = (short)(sl * W + j);
                }
                next_super += q.tiles / W;
            } else {
                if (open_super < 0 || open_fill + q.tiles > W) { open_super = next_super++; open_fill = 0; }
                for (int t = 0; t < q.tiles; ++t) {
                    p.super_tile[open_super * W + open_fill + t] = (short)(q.tile_base + t);
                    p.tile_slot[q.tile_base + t] = (short)(open_super * W + open_fill + t);
                }
                open_fill += q.tiles;
            }
        }
        if (next_super != n_super || (long)n_super * W > zp::MAX_TILES) return 1;
    }
    p.total = (long)n_super * p.S;
    // equal runs over all gangs; runs shorter than eight stages would be mostly set-up and drain
    const size_t seg_bytes = pair_segment_bytes(p.any_bias != 0);
    const size_t room = workspace && workspace_bytes > (size_t)kHeaderBytes ? workspace_bytes - kHeaderBytes : 0;
    const long max_segments = (long)(room / seg_bytes) / W;          // per gang position
    if (max_segments < n_super) return 1;
    long U = ceil_div(p.total, (long)(kNumPairs / W));
    if (U < 8) U = p.total < 8 ? p.total : 8;
    // a small workspace (the fixed array of the entry point without one) limits the number of runs
    while (zp::segment_of(p.total - 1, p.S, (int)U, (long)p.S / gcd_l(p.S, U) * U) + 1 > max_segments) {
        const long runs = ceil_div(p.total, U);
        if (runs <= 1) return 1;
        U = ceil_div(p.total, runs - 1);
    }
    p.U = (int)U;
    p.lcm = (long)p.S / gcd_l(p.S, U) * U;
    const long n_segments = (zp::segment_of(p.total - 1, p.S, p.U, p.lcm) + 1) * W;
    p.n_segments = n_segments;
    for (int t = 0; t < G; ++t) {                                   // the reduce kernel's view of the same cut
        const long sl = p.tile_slot[t] / W, j = p.tile_slot[t] % W;
        const long s0 = zp::segment_of(sl * p.S, p.S, p.U, p.lcm), s1 = zp::segment_of((sl + 1) * p.S - 1, p.S, p.U, p.lcm);
        p.seg_first[t] = (int)(s0 * W + j);
        p.seg_count[t] = (short)(s1 - s0 + 1);
    }
    for (int l = 0; l < n; ++l)
        for (int t = 0; t < p.layer[l].tiles; ++t) p.tile_layer[p.layer[l].tile_base + t] = (unsigned char)l;
    p.part = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes);
    p.bias_part = p.any_bias ? p.part + (size_t)n_segments * zp::SEG_ELEMS : nullptr;
    if (fuse_noise) {
        p.noise_scale = noise->scale;
        p.k0 = (uint32_t)noise->seed; p.k1 = (uint32_t)(noise->seed >> 32);
        if (noise_done) *noise_done = true;
    }
    const auto kernel = any_split ? tc::zta_pair_kernel<true, true> : cut ? tc::zta_pair_kernel<false, true> : tc::zta_pair_kernel<false, false>;
    if (!enable_smem(kernel, zp::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
    const int pairs = (int)ceil_div(p.total, U) * W;
    DPCLIP_LOGF("clipped sum, CTA pairs: %d layer(s), B*T=%ld, %d tiles of up to 512x256 in %d super-layer(s) of %d, %d stages per tile, "
                "%d pairs in gangs of %d, runs of %ld stages, %ld segments, noise %s", n, R, G, n_super, W, p.S, pairs, W, U,
                n_segments, fuse_noise ? "in the reduce" : "separate");
    int rc;
    if (take_overlap()) {
        rc = launch_behind(kernel, dim3(2 * pairs), zp::THREADS, zp::SMEM_BYTES, st, maps, p);
    } else {
        kernel<<<2 * pairs, zp::THREADS, zp::SMEM_BYTES, st>>>(maps, p);
        rc = launch_status();
    }
    if (rc) return rc;
    // one wave of CTAs (six of 256 threads and 40 registers per SM) over the 4-row blocks of all tiles
    long blocks = (long)G * (zp::BM / 4);
    if (blocks > 6L * kNumSMs) blocks = 6L * kNumSMs;
    // Behind the sums the reduce draws its first noise on SMs that have no pair, or beside the short drains of cut tiles; beside the full
    // drains of pairs on all SMs it holds these up.  Steps, behind / in order: one layer of 512 -> 512, 1024 rows 30.7 / 32.3 us, 8192 (32 pairs)
    // 37.7 / 38.9, 16384 (64 pairs) 41.1 / 38.9, 32768 (74 pairs) 59.3 / 53.5; 1024 -> 1024, 2048 rows (32 pairs) 38.9 / 40.6, 4096 (64) 45.0 /
    // 42.4, 8192 (72) 55.1 / 51.7; cut tiles, 128 -> 300, 32768 rows 46.0 / 47.2, a text model of 300 and 1100 features 90.3 / 91.2.
    constexpr int kPairsBeside = 56;                       // nothing measured between 48 and 64
    if (cut || pairs <= kPairsBeside) return launch_behind(tc::reduce_segments_kernel, dim3((unsigned)blocks), 256, 0, st, p);
    tc::reduce_segments_kernel<<<(unsigned)blocks, 256, 0, st>>>(p);
    return launch_status();
}

int launch_zta_tc(const void* A, long lda, const void* Z, long ldz, int B, int T, int d_in, int d_out,
                  bool norm_mode, int has_bias, const float* clip, float* gW, long ldg, float* gb, float* sq,
                  void* workspace, size_t workspace_bytes, const NoiseSpec* noise, bool* noise_done,
                  cudaStream_t st, bool fit_to_workspace = false, bool split = false) {
    namespace z = tc::zta;
    const long R = (long)B * T;
    int mt = d_out > 128 ? 2 : 1;
    if (path_switch(SW_TILE_M1)) mt = 1;
    if (path_switch(SW_TILE_M2)) mt = 2;
    const bool pair = !norm_mode && mt == 2 && pair_tile_ok(d_out);
    if (split && !norm_mode) mt = 1;            // the second operand plane leaves room for the small tile only
    const int bk = mt == 2 ? z::Cfg<2>::BK : z::Cfg<1>::BK;           // rows of a TMA box = rows of a stage
    z::Maps maps;
    if (!make_map_bf16(&maps.a[0], A, R, d_in, lda, 64, bk) || !make_map_bf16(&maps.z[0], Z, R, d_out, ldz, 64, bk))
        return DPCLIP_ERR_CUDA;
    z::Params p;
    memset(&p, 0, sizeof(p));
    p.R = (int)R; p.T = T; p.d_in = d_in; p.d_out = d_out;
    p.norm_mode = norm_mode ? 1 : 0;
    p.status = static_cast<int*>(workspace);
    if (norm_mode) {
        p.do_bias = has_bias ? 1 : 0;
        p.sq = sq;
    } else {
        p.clip = clip; p.gW = gW; p.ldg = ldg; p.gb = gb;
        p.do_bias = gb ? 1 : 0;
        p.vec_ok = aligned_to(gW, 16) && ldg % 4 == 0;
    }
    if (pair) {
        const StreamLayer one = {A, lda, Z, ldz, d_in, d_out, gW, ldg, gb, noise ? noise->sid_w : 0ull, noise ? noise->sid_b : 0ull, clip, split};
        const int rc = launch_zta_stream(&one, 1, B, T, noise, noise_done, workspace, workspace_bytes, st);
        if (rc <= 0) return rc;                 // 1: not even one segment per tile fits -> the single-CTA kernel below
    }
    if (mt == 2)
        return launch_zta_tc_mt<2>(maps, p, B, norm_mode, gW, ldg, gb, sq, d_in, d_out, workspace, workspace_bytes,
                                   noise, noise_done, st, fit_to_workspace);
    if (split && !norm_mode)
        return launch_zta_tc_mt<1, true>(maps, p, B, norm_mode, gW, ldg, gb, sq, d_in, d_out, workspace, workspace_bytes,
                                         noise, noise_done, st, fit_to_workspace);
    return launch_zta_tc_mt<1>(maps, p, B, norm_mode, gW, ldg, gb, sq, d_in, d_out, workspace, workspace_bytes,
                               noise, noise_done, st, fit_to_workspace);
}

// Clipped sums (+ noise) of n layers of ONE shape in one tensor-core launch and one reduce launch.
// Returns 1 when the group does not qualify (the caller then goes layer by layer).
int launch_zta_tc_group(const dpclip_layer* const* ls, const int* index, int n, int B, const float* clip,
                        float noise_scale, unsigned long long seed, unsigned long long stream_id0,
                        void* workspace, size_t workspace_bytes, cudaStream_t st, bool split = false) {
    namespace z = tc::zta;
    if (n < 2 || n > z::MAX_LAYERS) return 1;
    const dpclip_layer& y0 = *ls[0];
    const long R = (long)B * y0.T;
    const int bk = y0.d_out > 128 && !split ? z::Cfg<2>::BK : z::Cfg<1>::BK;
    z::Maps maps;
    GradGroup grp;
    memset(&grp, 0, sizeof(grp));
    grp.n = n;
    float* any_gb = nullptr;
    bool vec_ok = true;
    for (int l = 0; l < n; ++l) {
        const dpclip_layer& y = *ls[l];
        if (!make_map_bf16(&maps.a[l], y.A, R, y.d_in, y.lda, 64, bk) ||
            !make_map_bf16(&maps.z[l], y.Zbar, R, y.d_out, y.ldz, 64, bk))
            return DPCLIP_ERR_CUDA;
        grp.gW[l] = y.gW; grp.gb[l] = y.has_bias ? y.gb : nullptr;
        grp.sid_w[l] = stream_id0 + 2ull * index[l]; grp.sid_b[l] = grp.sid_w[l] + 1;
        if (grp.gb[l]) any_gb = grp.gb[l];
        vec_ok = vec_ok && aligned_to(y.gW, 16);
    }
    z::Params p;
    memset(&p, 0, sizeof(p));
    p.R = (int)R; p.T = y0.T; p.d_in = y0.d_in; p.d_out = y0.d_out;
    p.status = static_cast<int*>(workspace);
    p.clip = clip; p.gW = y0.gW; p.ldg = y0.d_in; p.gb = any_gb;
    p.do_bias = any_gb ? 1 : 0;
    p.vec_ok = vec_ok && y0.d_in % 4 == 0;
    const NoiseSpec ns = {noise_scale, seed, 0, 0};             // the streams come from the group
    bool noise_done = false;
    int rc;
    if (split)
        rc = launch_zta_tc_mt<1, true>(maps, p, B, false, y0.gW, y0.d_in, any_gb, nullptr, y0.d_in, y0.d_out, workspace,
                                       workspace_bytes, &ns, &noise_done, st, false, &grp);
    else if (y0.d_out > 128)
        rc = launch_zta_tc_mt<2>(maps, p, B, false, y0.gW, y0.d_in, any_gb, nullptr, y0.d_in, y0.d_out, workspace,
                                 workspace_bytes, &ns, &noise_done, st, false, &grp);
    else
        rc = launch_zta_tc_mt<1>(maps, p, B, false, y0.gW, y0.d_in, any_gb, nullptr, y0.d_in, y0.d_out, workspace,
                                 workspace_bytes, &ns, &noise_done, st, false, &grp);
    if (rc) return rc;
    if (noise_scale > 0.f && !noise_done) return DPCLIP_ERR_UNSUPPORTED;     // the outputs are dense
    return DPCLIP_OK;
}

// fp32 layers on the tensor cores (error-compensated tf32): TMA needs 16-byte aligned bases and rows
inline bool tf32_eligible(const void* A, long lda, const void* Z, long ldz, int B, int T, int d_in, int d_out,
                          dpclip_dtype dtype) {
    if (dtype != DPCLIP_F32) return false;
    if (path_switch(SW_FORCE_SIMT)) return false;
    if (!(aligned_to(A, 16) && aligned_to(Z, 16) && lda % 4 == 0 && ldz % 4 == 0)) return false;
    // worth it once there is real contraction work; tiny layers stay on the fp32-ALU kernels
    return (double)B * T * d_in * d_out >= 32.0 * 1024 * 1024;
}

bool make_map_f32(CUtensorMap* map, const void* base, long rows, long cols, long ld, int box_cols, int box_rows,
                  CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int launch_zta_tf32(const void* A, long lda, const void* Z, long ldz, int B, int T, int d_in, int d_out,
                    bool norm_mode, int has_bias, const float* clip, float* gW, long ldg, float* gb, float* sq,
                    void* workspace, size_t workspace_bytes, const NoiseSpec* noise, bool* noise_done,
                    cudaStream_t st, const tc::ConvGather* conv = nullptr) {
    namespace t = tc::t32;
    const long R = (long)B * T;
    CUtensorMap ma, mz;
    if (!make_map_f32(&mz, Z, R, d_out, ldz, 32, t::BK)) return DPCLIP_ERR_CUDA;
    if (conv) ma = mz;                                       // A is gathered from the feature map: no tensor map for it
    else if (!make_map_f32(&ma, A, R, d_in, lda, 32, t::BK)) return DPCLIP_ERR_CUDA;
    tc::zta::Params p;
    memset(&p, 0, sizeof(p));
    p.R = (int)R; p.T = T; p.d_in = d_in; p.d_out = d_out;
    p.norm_mode = norm_mode ? 1 : 0;
    p.status = static_cast<int*>(workspace);
    p.tiles_m = ceil_div(d_out, t::BM); p.tiles_n = ceil_div(d_in, t::BN);
    const int tiles = p.tiles_m * p.tiles_n;
    int ksplit = 1;
    if (norm_mode) {
        p.do_bias = has_bias ? 1 : 0;
        p.sq = sq;
        p.n_items = B * tiles;
        if (!clear_sq(sq, (size_t)B, st)) return DPCLIP_ERR_CUDA;
    } else {
        p.clip = clip; p.gW = gW; p.ldg = ldg; p.gb = gb;
        p.do_bias = gb ? 1 : 0;
        p.vec_ok = aligned_to(gW, 16) && ldg % 4 == 0;
        const int nkb = ceil_div(R, t::BK);
        // two accumulator buffers: two items per SM when they stay long enough, else one wave
        const int sms = sm_budget();
        const int per_sm = (tiles <= sms && nkb / ((2 * sms) / tiles) >= 16) ? 2 : 1;
        ksplit = (per_sm * sms) / tiles;
        if (ksplit > nkb) ksplit = nkb;
        if (ksplit < 1) ksplit = 1;
        p.kb_per_split = ceil_div(nkb, ksplit);
        ksplit = ceil_div(nkb, p.kb_per_split);
        p.n_items = tiles * ksplit;
        if (ksplit > 1) {
            const size_t part_bytes = (size_t)p.n_items * t::BM * t::BN * 4;
            const size_t bias_bytes = gb ? (size_t)p.n_items * t::BM * 4 : 0;
            if (workspace_bytes < kHeaderBytes + part_bytes + bias_bytes) return DPCLIP_ERR_WORKSPACE;
            p.part = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes);
            p.bias_part = gb ? p.part + part_bytes / 4 : nullptr;
        } else if (gb && cudaMemsetAsync(gb, 0, sizeof(float) * (size_t)d_out, st) != cudaSuccess) {
            return DPCLIP_ERR_CUDA;
        }
    }
    const int grid = p.n_items < sm_budget() ? p.n_items : sm_budget();
    if (conv) {
        if (!enable_smem(tc::zta_tf32_kernel<true>, t::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
        tc::zta_tf32_kernel<true><<<grid, t::THREADS, t::SMEM_BYTES, st>>>(ma, mz, p, *conv);
    } else {
        tc::ConvGather none;
        memset(&none, 0, sizeof(none));
        if (!enable_smem(tc::zta_tf32_kernel<false>, t::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
        tc::zta_tf32_kernel<false><<<grid, t::THREADS, t::SMEM_BYTES, st>>>(ma, mz, p, none);
    }
    int rc = launch_status();
    if (rc || norm_mode || ksplit == 1) return rc;
    return launch_reduce_partials(p, tiles, ksplit, t::BM, t::BN, d_in, d_out, gW, ldg, gb, noise, noise_done, st);
}

// ---------------------------------------------------------------------------
// Many layers in one launch on CTA pairs (kernels_group.cuh)
// ---------------------------------------------------------------------------
struct GroupLayer {
    const void* A; long lda; const void* Z; long ldz;
    int T, d_in, d_out;
    bool bias;
    float* sq;                                             // norms
    const float* clip;                                     // clipped sums
    float* gW; long ldg; float* gb; unsigned long long sid_w, sid_b;
};
constexpr size_t kGroupSlotBytes = tc::zg::SLOT_ELEMS * 4 + 256 * 4;
constexpr int kGroupMinRun = 4;                            // stages of a run, at least: shorter ones are mostly set-up and drain

// Tiling of a layer: which operand the M side is (256-column tiles), and the N side's tile width.
struct GroupTiling { bool z_on_m; int tiles_m, tiles_n, N; };
inline GroupTiling group_tiling(int d_in, int d_out) {
    auto make = [](bool z_on_m, int dm, int dn) {
        GroupTiling t;
        t.z_on_m = z_on_m;
        t.tiles_m = ceil_div(dm, tc::zg::BM);
        const int parts = ceil_div(dn, tc::zg::BN_MAX);
        t.N = ceil_div(ceil_div(dn, parts), 64) * 64;
        t.tiles_n = ceil_div(dn, t.N);
        return t;
    };
    // a stage costs about as much as its columns, 256 + N (bytes through shared memory); A on the M side when equal: its
    // partial tiles lie the way gW does
    const GroupTiling a = make(false, d_in, d_out), z = make(true, d_out, d_in);
    const long ca = (long)a.tiles_m * a.tiles_n * (256 + a.N), cz = (long)z.tiles_m * z.tiles_n * (256 + z.N);
    return cz < ca ? z : a;
}
// fp32: layers with a side of at most 128 leave the 256-column tiles mostly prepared for few products, and are as fast in
// zta_tf32_kernel (128 x 128 tiles), one or two of them; from three on the shared launch wins on one stream (three layers 288 -> 64,
// T = 256, 128 examples: 215 us a step by layer, 194 together; 576 -> 128, T = 64: 143 / 108; four 100 -> 100, T = 200, 64: 136 / 84).
inline bool group_wide(int d_in, int d_out) { return d_in > 128 && d_out > 128; }
constexpr int kGroupFrom = 3;
// On several streams the launches of zta_tf32_kernel run side by side, so a narrow layer joins only where the shared launch's
// extra work on it takes less than the launches it saves: microseconds over all SMs, a pair's stage 0.00225 a column, a CTA's
// 128 x 128 stage 0.7, a tile's drain 1 and 1.5, saved 1.1 per layer of the clipped sum and 2 in the norms.  Steps on four streams,
// by layer / sums together / norms together / both: three layers 288 -> 64, T = 256, 128 examples: 169 / 178 / 182 / 189;
// 576 -> 128, T = 64: 111 / 107 / 107 / 103; 512 -> 64, T = 256, 64: 131 / 121 / 124 / 113; four 100 -> 100, T = 200, 64:
// 70 / 66 / 80 / 78.
inline double group_stage_us(int d_in, int d_out) {
    const GroupTiling t = group_tiling(d_in, d_out);
    return t.tiles_m * t.tiles_n * (256 + t.N) * 0.00225;
}
inline bool group_joins(const dpclip_layer& y, int B, int n, bool norm) {
    if (group_wide(y.d_in, y.d_out)) return true;
    const GroupTiling t = group_tiling(y.d_in, y.d_out);
    const double pair = group_stage_us(y.d_in, y.d_out) / (kNumSMs / 2), tiles = ceil_div(y.d_out, 128) * ceil_div(y.d_in, 128);
    if (!norm) return ceil_div((long)B * y.T, 32L) * (pair - tiles * 0.7 / kNumSMs) <= 1.1 * n;
    const int stages = ceil_div(y.T, 32L);
    return B * (stages * pair + t.tiles_m * t.tiles_n / (kNumSMs / 2.0) - tiles * (stages * 0.7 + 1.5) / kNumSMs) <= 2.0;
}
inline int group_tiles(int d_in, int d_out) { const GroupTiling t = group_tiling(d_in, d_out); return t.tiles_m * t.tiles_n; }

// Clears the rows of sq that a launch accumulates into, adjacent rows in one memset.
inline int clear_rows(float* const* rows, int n, int B, cudaStream_t st) {
    int order[64];
    if (n > 64) return DPCLIP_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i) {
        int j = i;
        for (; j > 0 && rows[order[j - 1]] > rows[i]; --j) order[j] = order[j - 1];
        order[j] = i;
    }
    for (int i = 0; i < n;) {
        float* begin = rows[order[i]];
        float* end = begin + B;
        int j = i + 1;
        while (j < n && rows[order[j]] == end) { end += B; ++j; }
        if (!clear_sq(begin, (size_t)(end - begin), st)) return DPCLIP_ERR_CUDA;
        i = j;
    }
    return DPCLIP_OK;
}

template <bool NORM>
int launch_group_kernel(const tc::zg::Maps& maps, const tc::zg::Params& p, cudaStream_t st) {
    constexpr int smem = tc::zg::Cfg::SMEM_BYTES;
    if (!enable_smem(tc::zta_group_kernel<NORM>, smem)) return DPCLIP_ERR_CUDA;
    if (take_overlap()) return launch_behind(tc::zta_group_kernel<NORM>, dim3(2 * p.n_runs), tc::zg::THREADS, smem, st, maps, p);
    tc::zta_group_kernel<NORM><<<2 * p.n_runs, tc::zg::THREADS, smem, st>>>(maps, p);
    return launch_status();
}

// norms of long examples keep the sums between two drains in a slot per run
constexpr long kGroupMinSlots = 8;
bool group_long_norms(const GroupLayer* ls, int n) {
    for (int l = 0; l < n; ++l) if (ls[l].T > tc::zg::FLUSH * tc::zg::Cfg::BK) return true;
    return false;
}
bool group_norm_room(const GroupLayer* ls, int n, size_t workspace_bytes) {
    return !group_long_norms(ls, n) || workspace_bytes >= kHeaderBytes + kGroupMinSlots * kGroupSlotBytes;
}
// Norms (norm = true) or clipped sums with noise of n fp32 layers.  Returns DPCLIP_OK, a negative status, or 1 when the
// workspace cannot hold a few partial tiles (clipped sums, norms of more than FLUSH stages; nothing has been launched then).
int launch_group(const GroupLayer* ls, int n, int B, bool norm, const NoiseSpec* noise, bool* noise_done,
                 void* workspace, size_t workspace_bytes, cudaStream_t st, const tc::gram::FactorsTail* tail = nullptr) {
    namespace g = tc::zg;
    constexpr int bk = g::Cfg::BK;
    const int max_runs = sm_budget() / 2;
    const size_t room = workspace && workspace_bytes > (size_t)kHeaderBytes ? workspace_bytes - kHeaderBytes : 0;
    const long cap = (long)(room / kGroupSlotBytes);
    const bool long_norms = norm && group_long_norms(ls, n);
    if ((!norm || long_norms) && cap < kGroupMinSlots) return 1;
    bool fuse_noise = !norm && noise && noise->scale > 0.f;
    for (int l = 0; l < n && fuse_noise; ++l) fuse_noise = ls[l].ldg == ls[l].d_in;
    if (norm) {
        for (int l0 = 0; l0 < n; l0 += 64) {
            float* rows[64];
            const int k = n - l0 < 64 ? n - l0 : 64;
            for (int l = 0; l < k; ++l) rows[l] = ls[l0 + l].sq;
            const int rc = clear_rows(rows, k, B, st);
            if (rc) return rc;
        }
    }
    g::Maps maps;
    g::Params p;
    int next = 0, next_tile = 0;                            // layer and its tile the next launch begins with
    while (next < n) {
        memset(&p, 0, sizeof(p));
        p.status = static_cast<int*>(workspace);
        p.first_chunk = p.last_chunk = 1;
        // the slots of a launch: its tiles and its runs
        const int runs_cap = (norm && !long_norms) || cap >= 2L * max_runs ? max_runs : (int)(cap / 2);
        int tiles = 0;
        double cost[g::MAX_LAYERS], total = 0.0;
        long units[g::MAX_LAYERS], n_units = 0;
        while (next < n && p.n_layers < g::MAX_LAYERS) {
            const GroupLayer& y = ls[next];
            const GroupTiling t = group_tiling(y.d_in, y.d_out);
            const int all = t.tiles_m * t.tiles_n;
            int take = all - next_tile;
            if (!norm && tiles + take > cap - runs_cap) {
                if (p.n_layers > 0) break;                  // the next launch begins with this layer
                take = (int)(cap - runs_cap);
            }
            const int k = p.n_layers;
            g::Layer& q = p.layer[k];
            const long R = (long)B * y.T;
            const void* pm = t.z_on_m ? y.Z : y.A; const long lm = t.z_on_m ? y.ldz : y.lda;
            const void* pn = t.z_on_m ? y.A : y.Z; const long ln = t.z_on_m ? y.lda : y.ldz;
            q.T = y.T; q.R = (int)R;
            q.d_m = t.z_on_m ? y.d_out : y.d_in; q.d_n = t.z_on_m ? y.d_in : y.d_out; q.z_on_m = t.z_on_m ? 1 : 0;
            const CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_128B;
            if (!make_map_f32(&maps.m[k], pm, R, q.d_m, lm, 32, bk, sw) || !make_map_f32(&maps.n[k], pn, R, q.d_n, ln, 32, bk, sw))
                return DPCLIP_ERR_CUDA;
            q.tiles_m = t.tiles_m; q.tiles_n = t.tiles_n; q.N = t.N;
            q.nkb = ceil_div(norm ? (long)y.T : R, (long)bk);
            q.tile0 = next_tile; q.tiles = take; q.tile_base = tiles; q.unit_base = (int)n_units;
            q.do_bias = norm ? y.bias : y.gb != nullptr;
            q.clip = y.clip; q.sq = y.sq;
            q.gW = y.gW; q.gb = y.gb; q.ldg = y.ldg; q.vec_ok = aligned_to(y.gW, 16) && y.ldg % 4 == 0;
            q.sw0 = (uint32_t)y.sid_w; q.sw1 = (uint32_t)(y.sid_w >> 32);
            q.sb0 = (uint32_t)y.sid_b; q.sb1 = (uint32_t)(y.sid_b >> 32);
            q.blk_begin = p.n_blocks;
            if (!norm) p.n_blocks += take * 8 * (t.N / 32);
            units[k] = norm ? (long)B * all : (long)take * q.nkb;
            cost[k] = norm ? (double)q.nkb * (256 + t.N) + 256 : 256 + t.N;
            total += cost[k] * units[k]; n_units += units[k]; tiles += take;
            if (n_units > 0x3FFFFFFFL) return DPCLIP_ERR_UNSUPPORTED;
            ++p.n_layers;
            if (!norm && next_tile + take < all) {           // a chunk of a layer
                p.first_chunk = next_tile == 0; p.last_chunk = 0;
                next_tile += take;
                break;
            }
            if (next_tile > 0) { p.first_chunk = 0; next_tile = 0; ++next; break; }
            ++next;
        }
        long runs = norm ? n_units : n_units / kGroupMinRun;
        if (runs > runs_cap) runs = runs_cap;
        if (runs < 1) runs = 1;
        p.n_runs = (int)runs;
        // equal shares of the total cost, cut between units
        {
            int k = 0;
            double before = 0.0;                             // cost of the layers before k
            for (int r = 0; r <= p.n_runs; ++r) {
                const double at = total * r / p.n_runs;
                while (k + 1 < p.n_layers && before + cost[k] * units[k] <= at) { before += cost[k] * units[k]; ++k; }
                long u = p.layer[k].unit_base + (long)((at - before) / cost[k] + 0.5);
                if (r == p.n_runs || u > n_units) u = n_units;
                p.run_begin[r] = (int)u;
            }
        }
        p.n_slots = norm ? p.n_runs : tiles + p.n_runs;
        p.part = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes);
        p.bias_part = p.part + (size_t)p.n_slots * g::SLOT_ELEMS;
        if (fuse_noise) { p.noise_scale = noise->scale; p.k0 = (uint32_t)noise->seed; p.k1 = (uint32_t)(noise->seed >> 32); }
        if (tail && next >= n) {
            p.tail = *tail;
            p.tail.done = reinterpret_cast<unsigned int*>(static_cast<char*>(workspace) + kTailCounterOffset);
        }
        DPCLIP_LOGF("group %s: %d layer(s), %d tiles, %ld units, %d runs", norm ? "norms" : "clipped sums", p.n_layers, tiles,
                    n_units, p.n_runs);
        int rc = norm ? launch_group_kernel<true>(maps, p, st) : launch_group_kernel<false>(maps, p, st);
        if (rc) return rc;
        if (norm) continue;
        const int blocks = p.n_blocks < 8 * kNumSMs ? p.n_blocks : 8 * kNumSMs;
        // 48 CTAs of one 192 -> 256 layer stood on six SMs.  Steps, packed / spread (in order): 192 -> 256, 64 examples of 200 positions 60.0 /
        // 46.7 us (47.1); 256 -> 512, 32 of 300: 58.1 / 50.1 (51.0); 148 -> 412 with two of 148 -> 148, 61 of 48: 46.6 / 42.7 (42.8); seven
        // layers of 512 and 2048 features, 32 of 128 (1184 CTAs): 421.2 / 423.5.
        const int spread = blocks < 4 * kNumSMs ? spread_smem(blocks, sizeof(float) * 32 * 33) : 0;      // more fill the SMs anyway
        // one limit for all launches: a smaller one would fail the launch another thread is about to make
        if (!enable_smem(tc::reduce_group_kernel, spread_smem(1, sizeof(float) * 32 * 33))) return DPCLIP_ERR_CUDA;
        if ((rc = launch_behind(tc::reduce_group_kernel, dim3(blocks), 256, spread, st, p))) return rc;
    }
    if (fuse_noise && noise_done) *noise_done = true;
    return DPCLIP_OK;
}

// clipped sum of one layer, optionally with the noise folded into the last pass over the output
int clipped_grad_impl(const void* A, long lda, const void* Zbar, long ldz, int B, int T, int d_in, int d_out,
                      dpclip_dtype dtype, const float* clip, float* gW, long ldg, float* gb, void* workspace,
                      size_t workspace_bytes, const NoiseSpec* noise, bool* noise_done, cudaStream_t st,
                      bool split = false) {
    DPCLIP_LOGF("clipped_grad B=%d T=%d %d->%d %s: %s", B, T, d_in, d_out, dtype == DPCLIP_F32 ? "f32" : "bf16",
                tc_eligible(A, lda, Zbar, ldz, dtype) ? "tcgen05 bf16"
                : (tf32_eligible(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype) && !narrow_layer(T, d_in, d_out, gb != nullptr, lda, ldz))
                      ? "tcgen05 3xtf32" : "fp32-ALU / narrow kernels");
    if (tc_eligible(A, lda, Zbar, ldz, dtype))
        return launch_zta_tc(A, lda, Zbar, ldz, B, T, d_in, d_out, false, 0, clip, gW, ldg, gb, nullptr, workspace,
                             workspace_bytes, noise, noise_done, st, false, split);
    if (tf32_eligible(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype) && !narrow_layer(T, d_in, d_out, gb != nullptr, lda, ldz)) {
        if (group_wide(d_in, d_out)) {
            GroupLayer y = {A, lda, Zbar, ldz, T, d_in, d_out, false, nullptr, clip, gW, ldg, gb,
                            noise ? noise->sid_w : 0ull, noise ? noise->sid_b : 0ull};
            const int rc = launch_group(&y, 1, B, false, noise, noise_done, workspace, workspace_bytes, st);
            if (rc <= 0) return rc;
        }
        return launch_zta_tf32(A, lda, Zbar, ldz, B, T, d_in, d_out, false, 0, clip, gW, ldg, gb, nullptr, workspace,
                               workspace_bytes, noise, noise_done, st);
    }
    return launch_simt_grad(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype, clip, gW, ldg, gb, st, workspace,
                            workspace_bytes, noise, noise_done);
}


// Whole step in two launches for models made of T = 1 layers only (see kernels_fused_t1.cuh).
// Returns 1 when the fused path does not apply (the caller then takes the per-layer path).
// Second launch of the fused step on the tensor cores (fp32 models).  Every layer must either be addressable
// by TMA (16-byte aligned base and row stride); the zb of a thin layer (at most 16 outputs) need not be.  Returns 1 when the model
// does not qualify, so that the caller falls back to the fp32-ALU kernel.
// Alignment that TMA asks of one operand of the fused tensor-core kernels (16-byte base and row stride).
inline bool t1_tma_ok(const void* ptr, long ld, dpclip_dtype dtype) {
    return aligned_to(ptr, 16) && ld % (dtype == DPCLIP_BF16 ? 8 : 4) == 0;
}

template <typename T, bool QUADS>
int launch_fused_t1_tc(tc::f1::Params& q, bool one_launch, int grid, void* workspace, cudaStream_t st) {
    namespace f = tc::f1;
    if (one_launch) {
        // the whole step as one cooperative launch (its CTAs meet at a grid-wide barrier)
        q.grid_counter = reinterpret_cast<unsigned int*>(static_cast<char*>(workspace) + kGridCounterOffset);
        if (!enable_smem(tc::t1_all_grads_tf32_kernel<true, T, QUADS>, f::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(grid); cfg.blockDim = dim3(f::THREADS); cfg.dynamicSmemBytes = f::SMEM_BYTES; cfg.stream = st;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeCooperative; attr.val.cooperative = 1;
        cfg.attrs = &attr; cfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&cfg, tc::t1_all_grads_tf32_kernel<true, T, QUADS>, q) != cudaSuccess) {
            cudaGetLastError();
            return 1;                       // cannot be made resident at once: take the two-launch form
        }
        return launch_status();
    }
    if (!enable_smem(tc::t1_all_grads_tf32_kernel<false, T, QUADS>, f::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
    tc::t1_all_grads_tf32_kernel<false, T, QUADS><<<grid, f::THREADS, f::SMEM_BYTES, st>>>(q);
    return launch_status();
}

int launch_fused_t1_tf32(const FusedT1Params& base, bool one_launch, dpclip_dtype dtype, void* workspace,
                         size_t workspace_bytes, cudaStream_t st) {
    namespace f = tc::f1;
    if (path_switch(SW_NO_T1_TF32)) return 1;
    if (!workspace || workspace_bytes < kHeaderBytes) return 1;
    static_assert(sizeof(f::Params) <= 4096, "kernel parameter space");
    f::Params q;
    memset(&q, 0, sizeof(q));
    q.base = base;
    q.status = static_cast<int*>(workspace);
    const bool bf16 = dtype == DPCLIP_BF16;
    int items = 0, tc_layers = 0;
    bool quads = true;
    for (int l = 0; l < base.L; ++l) {
        const FusedT1Layer& y = base.layer[l];
        quads = quads && y.d_in % 4 == 0;
        const bool thin = y.d_out <= f::THIN_MAX_OUT;
        if (!t1_tma_ok(y.A, y.lda, dtype) || !(t1_tma_ok(y.Z, y.ldz, dtype) || thin)) return 1;
        q.item_begin[l] = items;
        q.thin[l] = thin ? 1 : 0;
        if (bf16) {
            if (!make_map_bf16(&q.map_a[l], y.A, base.B, y.d_in, y.lda, 64, f::BK)) return DPCLIP_ERR_CUDA;
            if (!thin && !make_map_bf16(&q.map_z[l], y.Z, base.B, y.d_out, y.ldz, 64, f::BK)) return DPCLIP_ERR_CUDA;
        } else {
            if (!make_map_f32(&q.map_a[l], y.A, base.B, y.d_in, y.lda, 32, f::BK)) return DPCLIP_ERR_CUDA;
            if (!thin && !make_map_f32(&q.map_z[l], y.Z, base.B, y.d_out, y.ldz, 32, f::BK)) return DPCLIP_ERR_CUDA;
        }
        q.tiles_n[l] = ceil_div(y.d_in, f::BN);
        items += ceil_div(y.d_out, f::BM) * q.tiles_n[l];
        if (!thin) ++tc_layers;
    }
    if (!tc_layers) return 1;
    q.total_items = items;
    const int grid = items < kNumSMs ? items : kNumSMs;
    if (bf16) return quads ? launch_fused_t1_tc<__nv_bfloat16, true>(q, one_launch, grid, workspace, st)
                           : launch_fused_t1_tc<__nv_bfloat16, false>(q, one_launch, grid, workspace, st);
    return quads ? launch_fused_t1_tc<float, true>(q, one_launch, grid, workspace, st)
                 : launch_fused_t1_tc<float, false>(q, one_launch, grid, workspace, st);
}

// Planes of a layer's operands in the workspace (kernels_t1_planes.cuh): c zb, and of fp32 models a too.
struct T1Planes { int pitch_z, pitch_a; size_t z, a; };
inline T1Planes t1_planes(int B, int d_in, int d_out, dpclip_dtype dtype) {
    const int planes = dtype == DPCLIP_F32 ? 3 : 1;
    T1Planes y;
    y.pitch_z = (int)round_up(d_out, 8); y.pitch_a = (int)round_up(d_in, 8);
    y.z = round_up((size_t)planes * B * y.pitch_z * 2, 256);
    y.a = dtype == DPCLIP_F32 ? round_up((size_t)planes * B * y.pitch_a * 2, 256) : 0;
    return y;
}
// Models of T = 1 layers that take the two launches of kernels_t1_planes.cuh: more than 16 output tiles of 128 x 128.  A step, one
// cooperative launch / two launches: fp32, 784-1000-1000-10, B = 128: 14.4 / 13.0 us, 1000-2000-1000, B = 64: 20.6 / 15.4, 512-512-512-10,
// B = 512: 30.8 / 23.2, 4096-4096-1000, B = 256: 121 / 78; bf16: the first 12.5 / 10.7, the last 72 / 46 (46 / 31 without noise).  784-256-10,
// B = 32 (16 tiles) would take 8.5 instead of 11.7, but up to there the one launch stays: it is the form whose barrier has its timeout
// tested, on that model.
inline bool t1_planes_pays(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype) {
    if (L <= 0 || L > FUSED_MAX_LAYERS || B > FUSED_MAX_B || path_switch(SW_NO_FUSED_T1 | SW_NO_T1_TF32 | SW_T1_TWO_LAUNCHES | SW_NO_T1_PLANES)) return false;
    long tiles = 0;
    for (int l = 0; l < L; ++l) {
        if (layers[l].T != 1 || layers[l].d_in <= 0 || layers[l].d_out <= 0) return false;
        tiles += (long)ceil_div(layers[l].d_out, (long)tc::t1p::BM) * ceil_div(layers[l].d_in, (long)tc::t1p::BN);
    }
    return tiles > 16 && tiles < 1L << 30;
}
inline size_t t1_planes_bytes(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype) {
    if (!t1_planes_pays(layers, L, B, dtype)) return 0;
    size_t n = 0;
    for (int l = 0; l < L; ++l) { const T1Planes y = t1_planes(B, layers[l].d_in, layers[l].d_out, dtype); n += y.z + y.a; }
    return n;
}

// 3-D bf16 matrix [planes][rows][cols], rows ld elements apart; rows and columns beyond a plane read as zero
bool make_map_planes(CUtensorMap* map, const void* base, int planes, long rows, long cols, long ld, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)ld * 2 * rows};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1}, estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename T>
int launch_t1_planes(const tc::t1p::Prep& prep, const tc::f1::Params& q, bool quads, int grid, cudaStream_t st) {
    namespace t = tc::t1p;
    constexpr int smem = t::Cfg<sizeof(T) == 4 ? 3 : 1>::SMEM_BYTES;
    const auto kernel = quads ? tc::t1_planes_kernel<T, true> : tc::t1_planes_kernel<T, false>;
    if (!enable_smem(kernel, smem)) return DPCLIP_ERR_CUDA;
    const bool few = prep.base.B <= t::PREP_FEW_EXAMPLES;
    const int rc = few ? launch_behind(tc::t1_prepare_kernel<T, 16>, dim3(prep.base.B), 512, 0, st, prep)
                       : launch_behind(tc::t1_prepare_kernel<T, 8>, dim3(prep.base.B), 256, 0, st, prep);
    return rc ? rc : launch_behind(kernel, dim3(grid), t::THREADS, smem, st, q);
}
// The whole step of a model of T = 1 layers.  1: the workspace lacks room, or the model is none for the tensor cores.
int try_t1_planes(const FusedT1Params& base, dpclip_dtype dtype, void* workspace, size_t workspace_bytes, cudaStream_t st) {
    namespace t = tc::t1p;
    const bool f32 = dtype == DPCLIP_F32;
    size_t at = kHeaderBytes;
    if (!workspace || !aligned_to(workspace, 16)) return 1;
    t::Prep prep;
    tc::f1::Params q;
    memset(&prep, 0, sizeof(prep)); memset(&q, 0, sizeof(q));
    prep.base = q.base = base;
    q.status = static_cast<int*>(workspace);
    bool quads = true, wide = false;
    for (int l = 0; l < base.L; ++l) {
        const FusedT1Layer& y = base.layer[l];
        // operands that the one-launch form does not take run on the fp32 ALUs, whose sums are of unrounded products
        const bool thin = y.d_out <= tc::f1::THIN_MAX_OUT;
        if (!t1_tma_ok(y.A, y.lda, dtype) || !(t1_tma_ok(y.Z, y.ldz, dtype) || thin)) return 1;
        wide = wide || !thin;
        const T1Planes s = t1_planes(base.B, y.d_in, y.d_out, dtype);
        prep.pitch_z[l] = s.pitch_z; prep.pitch_a[l] = s.pitch_a;
        prep.za[l] = reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + at); at += s.z;
        prep.aa[l] = reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + at); at += s.a;
        quads = quads && y.d_in % 4 == 0;
    }
    if (workspace_bytes < at || !wide) return 1;
    const int planes = f32 ? 3 : 1, bk = f32 ? t::Cfg<3>::BK : t::Cfg<1>::BK;
    int items = 0;
    for (int l = 0; l < base.L; ++l) {
        const FusedT1Layer& y = base.layer[l];
        if (!make_map_planes(&q.map_z[l], prep.za[l], planes, base.B, y.d_out, prep.pitch_z[l], bk) ||
            !(f32 ? make_map_planes(&q.map_a[l], prep.aa[l], planes, base.B, y.d_in, prep.pitch_a[l], bk)
                  : make_map_planes(&q.map_a[l], y.A, 1, base.B, y.d_in, y.lda, bk))) return DPCLIP_ERR_CUDA;
        q.item_begin[l] = items;
        q.tiles_n[l] = ceil_div(y.d_in, (long)t::BN);
        items += ceil_div(y.d_out, (long)t::BM) * q.tiles_n[l];
    }
    q.total_items = items;
    const int grid = items < kNumSMs ? items : kNumSMs;
    DPCLIP_LOGF("T = 1 model in two launches: %d layer(s), B=%d, %d tiles", base.L, base.B, items);
    return f32 ? launch_t1_planes<float>(prep, q, quads, grid, st) : launch_t1_planes<__nv_bfloat16>(prep, q, quads, grid, st);
}

// One T = 1 layer of the caller's model as the fused kernels see it.  Returns 0, 1 (the layer does not
// qualify for the fused kernels) or a negative argument error.
int fill_fused_t1_layer(FusedT1Layer& f, const dpclip_layer& y, int index, int B, dpclip_dtype dtype, int tile,
                        int& tiles) {
    if (y.T != 1 || y.ldg != y.d_in) return 1;
    if (y.method != DPCLIP_AUTO && y.method != DPCLIP_T1) return 1;
    int rc = check_layer_args(y.A, y.lda, y.Zbar, y.ldz, B, 1, y.d_in, y.d_out, dtype);
    if (rc) return rc;
    if (!y.gW || (y.has_bias && !y.gb)) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(y.gW, 16) || (y.gb && !aligned_to(y.gb, 4))) return 1;
    f.A = y.A; f.lda = y.lda; f.Z = y.Zbar; f.ldz = y.ldz;
    f.d_in = y.d_in; f.d_out = y.d_out; f.has_bias = y.has_bias ? 1 : 0;
    f.vec_a = vec4_ok(y.A, y.lda, dtype); f.vec_z = vec4_ok(y.Zbar, y.ldz, dtype);
    f.gW = y.gW; f.gb = y.has_bias ? y.gb : nullptr;
    f.tiles_m = ceil_div(y.d_out, tile); f.tiles_n = ceil_div(y.d_in + f.has_bias, tile);
    f.tile_begin = tiles;
    f.index = index;
    tiles += f.tiles_m * f.tiles_n;
    return 0;
}

// The T = 1 layers of a model that also has T > 1 layers (fp32): their norms in one launch (into their rows
// of sq), and, once the factors of the whole model exist, their clipped sums with noise in one tensor-core
// launch.  `group` lists the layers' positions in the model.  prepare returns 0 when the group qualifies.
struct T1Group {
    FusedT1Params p;
    bool active = false;
};

int prepare_t1_group(T1Group& g, const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                     unsigned long long seed, unsigned long long stream_id0, float* sq, const float* clip,
                     bool mixed_only = true) {
    g.active = false;
    if (B > FUSED_MAX_B) return 0;
    if (path_switch(SW_NO_FUSED_T1)) return 0;
    if (path_switch(SW_NO_T1_TF32)) return 0;
    memset(&g.p, 0, sizeof(g.p));
    int n = 0, tiles = 0, wide = 0;
    for (int l = 0; l < L; ++l) {
        if (layers[l].T != 1) continue;
        if (n == FUSED_MAX_LAYERS) return 0;
        const int rc = fill_fused_t1_layer(g.p.layer[n], layers[l], l, B, dtype, 64, tiles);
        if (rc < 0) return rc;
        if (rc) return 0;
        const FusedT1Layer& y = g.p.layer[n];
        if (!t1_tma_ok(y.A, y.lda, dtype) || !(t1_tma_ok(y.Z, y.ldz, dtype) || y.d_out <= tc::f1::THIN_MAX_OUT))
            return 0;
        if (y.d_out > tc::f1::THIN_MAX_OUT) ++wide;
        ++n;
    }
    if (n == 0 || wide == 0 || (mixed_only && n == L)) return 0;    // the kernel wants one tensor-core layer
    g.p.L = n; g.p.B = B; g.p.total_tiles = tiles;
    g.p.C = C; g.p.noise_scale = sigma * C;
    g.p.k0 = (uint32_t)seed; g.p.k1 = (uint32_t)(seed >> 32); g.p.stream_id0 = stream_id0;
    g.p.sq = sq; g.p.clip = nullptr; g.p.norms = nullptr; g.p.clip_in = clip;
    g.active = true;
    return 0;
}

int try_fused_t1_step(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                      unsigned long long seed, unsigned long long stream_id0, float* sq, float* clip,
                      float* norms, void* workspace, size_t workspace_bytes, cudaStream_t st) {
    if (L > FUSED_MAX_LAYERS || B > FUSED_MAX_B) return 1;
    if (path_switch(SW_NO_FUSED_T1)) return 1;
    FusedT1Params p;
    memset(&p, 0, sizeof(p));
    // fp32-ALU form: 64 x 64 tiles, several CTAs per SM hide the global-load latency of these short (K = B)
    // products (128 x 128 register tiles, one CTA per SM, measured slower: 61 vs 39 us per step on the
    // 784-1000-1000-10, B = 128 model).
    const int tile = 64;
    int tiles = 0;
    for (int l = 0; l < L; ++l) {
        const int rc = fill_fused_t1_layer(p.layer[l], layers[l], l, B, dtype, tile, tiles);
        if (rc) return rc;
    }
    p.L = L; p.B = B; p.total_tiles = tiles;
    p.C = C; p.noise_scale = sigma * C;
    p.k0 = (uint32_t)seed; p.k1 = (uint32_t)(seed >> 32); p.stream_id0 = stream_id0;
    p.sq = sq; p.clip = clip; p.norms = norms;
    const int rows = L * B;
    const int grid_n = rows;
    const int grid_g = tiles < 4 * kNumSMs ? tiles : 4 * kNumSMs;
    const int smem64 = FusedT1Cfg<64>::SMEM_BYTES;
    if (t1_planes_pays(layers, L, B, dtype)) {
        const int rc = try_t1_planes(p, dtype, workspace, workspace_bytes, st);
        if (rc <= 0) return rc;
    }
    bool one = true;
    if (path_switch(SW_T1_TWO_LAUNCHES)) one = false;
    if (one) {
        const int rc = launch_fused_t1_tf32(p, true, dtype, workspace, workspace_bytes, st);
        if (rc <= 0) return rc;
    }
    if (dtype == DPCLIP_F32) t1_all_norms_kernel<float><<<grid_n, 128, 0, st>>>(p);
    else t1_all_norms_kernel<__nv_bfloat16><<<grid_n, 128, 0, st>>>(p);
    if (launch_status()) return DPCLIP_ERR_CUDA;
    const int rc = launch_fused_t1_tf32(p, false, dtype, workspace, workspace_bytes, st);
    if (rc <= 0) return rc;
    if (dtype == DPCLIP_F32) t1_all_grads_kernel<float, 64><<<grid_g, SIMT_THREADS, smem64, st>>>(p);
    else t1_all_grads_kernel<__nv_bfloat16, 64><<<grid_g, SIMT_THREADS, smem64, st>>>(p);
    return launch_status();
}

}  // namespace

extern "C" {

int dpclip_version(void) { return 100; }
int dpclip_debug_build(void) {
#ifdef DPCLIP_DEBUG
    return 1;
#else
    return 0;
#endif
}

// An empty kernel with the launch shape of the one-launch T = 1 step: what a launch costs before it computes.
__global__ void null_launch_kernel(int* sink) { if (sink && threadIdx.x == 0xFFFFFF) *sink = 0; }

int dpclip_null_launch(int cooperative, int grid, void* stream) {
    namespace f = tc::f1;
    if (grid < 1 || grid > kNumSMs) return DPCLIP_ERR_INVALID_ARG;
    if (!enable_smem(null_launch_kernel, f::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(f::THREADS); cfg.dynamicSmemBytes = f::SMEM_BYTES;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative; attr.val.cooperative = cooperative ? 1 : 0;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    int* none = nullptr;
    if (cudaLaunchKernelEx(&cfg, null_launch_kernel, none) != cudaSuccess) { cudaGetLastError(); return DPCLIP_ERR_CUDA; }
    return launch_status();
}

unsigned long long dpclip_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }
void dpclip_reload_path_switches(void) { read_path_switches(); }

#ifdef DPCLIP_TRACE
int dpclip_trace_copy(unsigned long long* host) {
    return cudaMemcpyFromSymbol(host, tc::g_trace, sizeof(unsigned long long) * 148 * 4 * 256) == cudaSuccess ? 0 : -5;
}
#endif

const char* dpclip_status_string(int status) {
    switch (status) {
        case DPCLIP_OK: return "ok";
        case DPCLIP_ERR_INVALID_ARG: return "invalid argument";
        case DPCLIP_ERR_UNSUPPORTED: return "method not supported for this dtype/shape/alignment";
        case DPCLIP_ERR_MISALIGNED: return "pointer not aligned to its element size";
        case DPCLIP_ERR_WORKSPACE: return "workspace missing or too small";
        case DPCLIP_ERR_CUDA: return "CUDA call or kernel launch failed";
        case DPCLIP_ERR_TIMEOUT: return "a bounded device-side wait ran out";
        case DPCLIP_ERR_RANGE: return "range-checked build: an index left its buffer (access skipped)";
        default: return "unknown status";
    }
}

int dpclip_pick_method(int B, int T, int d_in, int d_out, long lda, long ldz, dpclip_dtype dtype) {
    (void)B;
    if (T == 1) return DPCLIP_T1;
    // alignment of the base pointers is not known here; rows must be 16-byte multiples for TMA
    if (dtype == DPCLIP_BF16 && lda % 8 == 0 && ldz % 8 == 0) {
        if (!path_switch(SW_FORCE_SIMT)) {
            const double gram = (double)T * (T + 1.0) * ((double)d_in + d_out);      // symmetric Gram blocks
            const double mat = 2.0 * T * (double)d_in * d_out;                       // one Zb_i^T A_i product
            return gram <= mat ? DPCLIP_GRAM : DPCLIP_MATERIALIZE;
        }
    }
    // fp32: materialised tiles on the tensor cores (error-compensated tf32) once the layer is large
    // enough and its rows are 16-byte multiples; narrow and small layers stay on the fp32 ALUs
    if (dtype == DPCLIP_F32 && lda % 4 == 0 && ldz % 4 == 0 && !narrow_layer(T, d_in, d_out, 1, lda, ldz) &&
        (double)B * T * d_in * d_out >= 32.0 * 1024 * 1024) {
        if (!path_switch(SW_FORCE_SIMT)) return DPCLIP_MATERIALIZE;
    }
    return DPCLIP_SIMT;
}

// The least workspace an entry point accepts for a layer (the public query may ask for more: see there).
static size_t workspace_floor(int B, int T, int d_in, int d_out, dpclip_dtype dtype) {
    if (dtype == DPCLIP_BF16) return kHeaderBytes + kTcScratchBytes;
    if ((double)B * T * d_in * d_out >= 32.0 * 1024 * 1024) return kHeaderBytes + kTcScratchBytes;
    return (size_t)kHeaderBytes;
}

size_t dpclip_workspace_bytes(int B, int T, int d_in, int d_out, dpclip_dtype dtype, dpclip_method method) {
    (void)method;
    // Layers that may take a tensor-core clipped sum (all bf16 layers; fp32 layers above the size where
    // the tf32 path is used) split their rows over CTAs and keep one partial tile per CTA in the
    // workspace; the bound does not depend on the layer's shape.
    if (dtype == DPCLIP_BF16) {
        // ... except for long layers whose tiles do not fill one wave of SMs: room for their preferred split
        size_t need = kTcScratchBytes;
        if (d_out > 128 && B > 0 && T > 0 && d_in > 0) {
            const int tiles = ceil_div(d_out, 256) * ceil_div(d_in, 256);
            const ZtaSplit split = zta_pick_split(ceil_div((long)B * T, 64L), tiles, 1);
            const size_t pref = zta_scratch_bytes(tiles, split.preferred, 256, true);
            if (split.preferred != split.one_wave && pref > need) need = pref;
            if (pair_tile_ok(d_out)) {                 // the CTA-pair kernel: one segment per tile and one per pair
                const size_t pneed = pair_scratch_bytes(pair_tiles(d_in, d_out));
                if (pneed > need) need = pneed;
            }
        }
        return kHeaderBytes + need;
    }
    if ((double)B * T * d_in * d_out >= 32.0 * 1024 * 1024) return kHeaderBytes + kTcScratchBytes;
    return (size_t)kHeaderBytes;
}

// Scratch for a step over these layers (not the staged copies: see stage_plan).
static size_t step_scratch_bytes(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype) {
    size_t ws = kHeaderBytes;
    if (!layers || L <= 0 || B <= 0) return ws;
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        if (y.T <= 0) continue;
        const size_t w = dpclip_workspace_bytes(B, y.T, y.d_in, y.d_out, dtype, (dpclip_method)y.method);
        if (w > ws) ws = w;
    }
    // the layers that share a clipped-sum launch of launch_group: a slot per tile of all of them and one per run
    {
        long tiles = 0;
        for (int l = 0; l < L; ++l) {
            const dpclip_layer& y = layers[l];
            if (y.T > 1 && y.d_in > 0 && y.d_out > 0 && dtype == DPCLIP_F32) tiles += group_tiles(y.d_in, y.d_out);
        }
        if (tiles > 512) tiles = 512;                        // more go in several launches
        const size_t need = kHeaderBytes + (size_t)(tiles + kNumPairs) * kGroupSlotBytes;
        if (tiles > 0 && need > ws && ws > (size_t)kHeaderBytes) ws = need;
    }
    if (const size_t planes = t1_planes_bytes(layers, L, B, dtype)) if (kHeaderBytes + planes > ws) ws = kHeaderBytes + planes;
    if (dtype != DPCLIP_BF16 || path_switch(SW_NO_GRAD_GROUP)) return ws;
    // layers of one T that share a CTA-pair launch (up to eight): one segment per tile of all of them + one per pair
    for (int l0 = 0; l0 < L; ++l0) {
        const dpclip_layer& y0 = layers[l0];
        if (y0.T <= 1 || !pair_shared_ok(y0.d_in, y0.d_out, (long)B * y0.T)) continue;
        bool first = true;
        for (int l = 0; l < l0; ++l) first = first && !(layers[l].T == y0.T && pair_shared_ok(layers[l].d_in, layers[l].d_out, (long)B * y0.T));
        if (!first) continue;
        int n = 0, tiles = 0;
        for (int l = l0; l < L; ++l) {
            if (layers[l].T != y0.T || !pair_shared_ok(layers[l].d_in, layers[l].d_out, (long)B * y0.T)) continue;
            tiles += pair_tiles(layers[l].d_in, layers[l].d_out);
            if (++n == tc::ztp::MAX_LAYERS) {
                if (kHeaderBytes + pair_scratch_bytes(tiles) > ws) ws = kHeaderBytes + pair_scratch_bytes(tiles);
                n = 0; tiles = 0;
            }
        }
        if (n >= 2 && kHeaderBytes + pair_scratch_bytes(tiles) > ws) ws = kHeaderBytes + pair_scratch_bytes(tiles);
    }
    return ws;
}

static size_t staged_workspace_bytes(const dpclip_layer* layers, const dpclip_model_layer* other, int L, int B, dpclip_dtype dtype,
                                     bool with_copies);

size_t dpclip_step_workspace_bytes(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype) {
    const size_t ws = step_scratch_bytes(layers, L, B, dtype);
    const size_t staged = staged_workspace_bytes(layers, nullptr, L, B, dtype, true);
    return staged > ws ? staged : ws;
}
size_t dpclip_step_side_workspace_bytes(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype) {
    const size_t ws = step_scratch_bytes(layers, L, B, dtype);
    const size_t staged = staged_workspace_bytes(layers, nullptr, L, B, dtype, false);
    return staged > ws ? staged : ws;
}

int dpclip_workspace_init(void* workspace, size_t workspace_bytes, void* stream) {
    if (!workspace || workspace_bytes < (size_t)kHeaderBytes) return DPCLIP_ERR_WORKSPACE;
    return cudaMemsetAsync(workspace, 0, kHeaderBytes, (cudaStream_t)stream) == cudaSuccess ? DPCLIP_OK
                                                                                             : DPCLIP_ERR_CUDA;
}

int dpclip_read_status(const void* workspace, int* host_status, void* stream) {
    if (!workspace || !host_status) return DPCLIP_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemcpyAsync(host_status, workspace, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return DPCLIP_ERR_CUDA;
    return cudaStreamSynchronize(st) == cudaSuccess ? DPCLIP_OK : DPCLIP_ERR_CUDA;
}

int dpclip_layer_sqnorms(const void* A, long lda, const void* Zbar, long ldz, int B, int T, int d_in,
                         int d_out, dpclip_dtype dtype, int has_bias, dpclip_method method, float* sq_layer,
                         void* workspace, size_t workspace_bytes, void* stream) {
    int rc = check_layer_args(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype);
    if (rc) return rc;
    if (!sq_layer) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(sq_layer, 4)) return DPCLIP_ERR_MISALIGNED;
    if (method == DPCLIP_AUTO) {
        method = (dpclip_method)dpclip_pick_method(B, T, d_in, d_out, lda, ldz, dtype);
        if (dtype == DPCLIP_BF16 && (method == DPCLIP_GRAM || method == DPCLIP_MATERIALIZE) &&
            !tc_eligible(A, lda, Zbar, ldz, dtype))
            method = DPCLIP_SIMT;
        if (dtype == DPCLIP_F32 && method == DPCLIP_MATERIALIZE && !tf32_eligible(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype))
            method = DPCLIP_SIMT;
    }
    if (!workspace || workspace_bytes < workspace_floor(B, T, d_in, d_out, dtype))
        return DPCLIP_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    DPCLIP_LOGF("layer_sqnorms B=%d T=%d %d->%d %s bias=%d: %s", B, T, d_in, d_out, dtype == DPCLIP_F32 ? "f32" : "bf16",
                has_bias, method == DPCLIP_T1 ? "T1 closed form" : method == DPCLIP_SIMT ? "materialise, fp32-ALU / narrow kernels"
                : method == DPCLIP_GRAM ? "Gram, tcgen05" : "materialise, tcgen05");
    switch (method) {
        case DPCLIP_T1:
            if (T != 1) return DPCLIP_ERR_UNSUPPORTED;
            return launch_t1_norms(A, lda, Zbar, ldz, B, d_in, d_out, dtype, has_bias, sq_layer, st);
        case DPCLIP_SIMT:
            return launch_simt_norms(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype, has_bias, sq_layer, st,
                                     static_cast<int*>(workspace));
        case DPCLIP_GRAM:
        case DPCLIP_MATERIALIZE:
            if (dtype == DPCLIP_F32) {                    // fp32: materialised tiles via error-compensated tf32
                if (method != DPCLIP_MATERIALIZE || !aligned_to(A, 16) || !aligned_to(Zbar, 16) || lda % 4 || ldz % 4)
                    return DPCLIP_ERR_UNSUPPORTED;
                if (group_wide(d_in, d_out)) {
                    GroupLayer y = {A, lda, Zbar, ldz, T, d_in, d_out, has_bias != 0, sq_layer};
                    rc = launch_group(&y, 1, B, true, nullptr, nullptr, workspace, workspace_bytes, st);
                    if (rc <= 0) return rc;              // 1: small layers come with the header alone
                }
                return launch_zta_tf32(A, lda, Zbar, ldz, B, T, d_in, d_out, true, has_bias, nullptr, nullptr, 0,
                                       nullptr, sq_layer, workspace, workspace_bytes, nullptr, nullptr, st);
            }
            if (!aligned_to(A, 16) || !aligned_to(Zbar, 16) || lda % 8 || ldz % 8)
                return DPCLIP_ERR_UNSUPPORTED;
            if (method == DPCLIP_GRAM)
                return launch_gram_norms(A, lda, Zbar, ldz, B, T, d_in, d_out, has_bias, sq_layer,
                                         (int*)workspace, st);
            return launch_zta_tc(A, lda, Zbar, ldz, B, T, d_in, d_out, true, has_bias, nullptr, nullptr, 0,
                                 nullptr, sq_layer, workspace, workspace_bytes, nullptr, nullptr, st);
        default:
            return DPCLIP_ERR_INVALID_ARG;
    }
}

static int gram_layers_sqnorms(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float* sq_layers,
                               int* taken, void* workspace, size_t workspace_bytes, void* stream,
                               const tc::gram::FactorsTail* tail, bool* tail_done);

int dpclip_gram_layers_sqnorms(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float* sq_layers,
                               int* taken, void* workspace, size_t workspace_bytes, void* stream) {
    return gram_layers_sqnorms(layers, L, B, dtype, sq_layers, taken, workspace, workspace_bytes, stream, nullptr, nullptr);
}

// tail: factors in the tail of the launch -- only when ONE launch takes every layer (all L rows of sq come from
// it); *tail_done says whether that happened.
static int gram_layers_sqnorms(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float* sq_layers,
                               int* taken, void* workspace, size_t workspace_bytes, void* stream,
                               const tc::gram::FactorsTail* tail, bool* tail_done) {
    if (tail_done) *tail_done = false;
    if (!layers || L <= 0 || B <= 0 || !sq_layers) return DPCLIP_ERR_INVALID_ARG;
    if (taken) for (int l = 0; l < L; ++l) taken[l] = 0;
    if (dtype != DPCLIP_BF16 || !workspace || workspace_bytes < (size_t)kHeaderBytes) return DPCLIP_OK;
    if (path_switch(SW_NO_GRAM_GROUP)) return DPCLIP_OK;
    namespace g = tc::gram;
    // One launch per kernel class (see gram_class); layers of class 1 join those of class 2 when there are any: a launch of their own
    // ends in a wave of its own (convolutions of 784 and 196 positions, 16 examples: two launches 8 and 17 us one after the other,
    // together 17).
    auto takes = [&](const dpclip_layer& y) {
        if (y.T <= 1 || check_layer_args(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype)) return false;
        if (!tc_eligible(y.A, y.lda, y.Zbar, y.ldz, dtype)) return false;
        const int method = y.method == DPCLIP_AUTO ? dpclip_pick_method(B, y.T, y.d_in, y.d_out, y.lda, y.ldz, dtype) : y.method;
        return method == DPCLIP_GRAM;
    };
    // the numbers of positions that occur, the widest layers of each and the order of their row blocks; a thirteenth is flattened
    struct { int T, n, width[g::MAX_LAYERS]; bool per_ex; } seen[12] = {};
    int n_seen = 0;
    bool more = false;
    auto of = [&](int T) { int k = 0; while (k < n_seen && seen[k].T != T) ++k; return k; };
    for (int l = 0; l < L; ++l) {
        if (!takes(layers[l])) continue;
        const int k = of(layers[l].T), w = layers[l].d_in + layers[l].d_out;
        if (k == n_seen) {
            if (n_seen == 12) { more = true; continue; }
            seen[n_seen++].T = layers[l].T;
        }
        auto& y = seen[k];
        int i = y.n < g::MAX_LAYERS ? y.n++ : w > y.width[g::MAX_LAYERS - 1] ? g::MAX_LAYERS - 1 : g::MAX_LAYERS;
        if (i == g::MAX_LAYERS) continue;
        for (; i > 0 && y.width[i - 1] < w; --i) y.width[i] = y.width[i - 1];
        y.width[i] = w;
    }
    bool any_long = more;
    for (int k = 0; k < n_seen; ++k) {
        seen[k].per_ex = gram_per_ex(seen[k].T, B, seen[k].width, seen[k].n);
        any_long = any_long || gram_class(seen[k].T, seen[k].per_ex) == 2;
    }
    auto per_ex_of = [&](int T) { const int k = of(T); return k < n_seen && seen[k].per_ex; };
    auto class_of = [&](int T) { const int c = gram_class(T, per_ex_of(T)); return c == 1 && any_long ? 2 : c; };
    for (int cls = 0; cls < 3; ++cls) {
        GramLayer batch[g::MAX_LAYERS];
        int idx[g::MAX_LAYERS];
        int n = 0;
        auto flush = [&]() -> int {
            // a single layer gains nothing from this entry point: leave it to the per-layer call
            if (n >= 2) {
                const bool with_tail = tail && n == L;             // this launch writes every row of sq
                const int rc = launch_gram_group(batch, n, cls, (int*)workspace, (cudaStream_t)stream, with_tail ? tail : nullptr);
                if (rc) return rc;
                if (taken) for (int i = 0; i < n; ++i) taken[idx[i]] = 1;
                if (with_tail && tail_done) *tail_done = true;
            }
            n = 0;
            return DPCLIP_OK;
        };
        for (int l = 0; l < L; ++l) {
            const dpclip_layer& y = layers[l];
            if (!takes(y) || class_of(y.T) != cls) continue;
            batch[n] = {y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, y.has_bias ? 1 : 0, sq_layers + (size_t)l * B,
                        per_ex_of(y.T)};
            idx[n] = l;
            if (++n == g::MAX_LAYERS) { const int rc = flush(); if (rc) return rc; }
        }
        const int rc = flush();
        if (rc) return rc;
    }
    return DPCLIP_OK;
}

static int shared_clipped_grad_launches(const dpclip_layer* layers, const bool* split, bool join, int L, int B, dpclip_dtype dtype,
                                        const float* clip, long clip_ld, float C, float sigma, unsigned long long seed,
                                        unsigned long long stream_id0, int* taken, void* workspace,
                                        size_t workspace_bytes, void* stream);

int dpclip_same_shape_layers_clipped_grad_noise(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype,
                                                const float* clip, float C, float sigma, unsigned long long seed,
                                                unsigned long long stream_id0, int* taken, void* workspace,
                                                size_t workspace_bytes, void* stream) {
    return shared_clipped_grad_launches(layers, nullptr, false, L, B, dtype, clip, 0, C, sigma, seed, stream_id0, taken, workspace,
                                        workspace_bytes, stream);
}

// join: take the layers of pair_shared_ok, not only those wide enough for the pair kernel by themselves.
// clip_ld = 0: one factor vector for all layers (global clipping); clip_ld > 0: layer l's factors are row l of
// clip[L][clip_ld] (per-layer clipping) -- then only the CTA-pair launches, which take a vector per layer, are made.
static int shared_clipped_grad_launches(const dpclip_layer* layers, const bool* split, bool join, int L, int B, dpclip_dtype dtype,
                                        const float* clip, long clip_ld, float C, float sigma, unsigned long long seed,
                                        unsigned long long stream_id0, int* taken, void* workspace,
                                        size_t workspace_bytes, void* stream) {
    if (!layers || L <= 0 || B <= 0) return DPCLIP_ERR_INVALID_ARG;
    if (!(C >= 0.f) || !(sigma >= 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (taken) for (int l = 0; l < L; ++l) taken[l] = 0;
    if (dtype != DPCLIP_BF16 || !workspace || workspace_bytes < (size_t)kHeaderBytes) return DPCLIP_OK;
    if (path_switch(SW_NO_GRAD_GROUP)) return DPCLIP_OK;
    namespace z = tc::zta;
    constexpr int kMaxTracked = 256;
    if (L > kMaxTracked) return DPCLIP_OK;
    bool done[kMaxTracked] = {false};
    auto candidate = [&](const dpclip_layer& y) {
        if (y.T <= 1 || !y.gW || y.ldg != y.d_in || (y.has_bias && !y.gb)) return false;
        if (check_layer_args(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype)) return false;
        if (!aligned_to(y.gW, 4) || (y.has_bias && !aligned_to(y.gb, 4))) return false;
        return tc_eligible(y.A, y.lda, y.Zbar, y.ldz, dtype);
    };
    // Layers wide enough for the CTA-pair kernel need not have one shape: all that have one T (hence the same
    // rows B*T) go into one stream-K launch, up to eight at a time.
    for (int l0 = 0; l0 < L; ++l0) {
        auto on_pairs = [&](const dpclip_layer& y) { return join ? pair_shared_ok(y.d_in, y.d_out, (long)B * y.T) : pair_tile_ok(y.d_out); };
        if (done[l0] || !candidate(layers[l0]) || !on_pairs(layers[l0])) continue;
        StreamLayer grp[tc::ztp::MAX_LAYERS];
        int idx[tc::ztp::MAX_LAYERS];
        int n = 0, tiles = 0;
        for (int l = l0; l < L && n < tc::ztp::MAX_LAYERS; ++l) {
            const dpclip_layer& y = layers[l];
            if (done[l] || y.T != layers[l0].T || !on_pairs(y) || !candidate(y)) continue;
            grp[n] = {y.A, y.lda, y.Zbar, y.ldz, y.d_in, y.d_out, y.gW, y.ldg, y.has_bias ? y.gb : nullptr,
                      stream_id0 + 2ull * l, stream_id0 + 2ull * l + 1, clip ? clip + (size_t)l * clip_ld : nullptr,
                      split && split[l]};
            idx[n] = l; ++n;
            tiles += pair_tiles(y.d_in, y.d_out);
        }
        if (n < 2) continue;                       // a single layer takes the same kernel through its own call
        // with less workspace than one segment per tile and pair the launch would run on fewer pairs: leave the
        // layers to their own launches then
        if (workspace_bytes < kHeaderBytes + pair_scratch_bytes(tiles)) continue;
        const NoiseSpec ns = {sigma * C, seed, 0, 0};
        bool noise_done = false;
        const int rc = launch_zta_stream(grp, n, B, layers[l0].T, &ns, &noise_done, workspace, workspace_bytes,
                                         (cudaStream_t)stream);
        if (rc < 0) return rc;
        if (rc > 0) continue;
        if (sigma * C > 0.f && !noise_done) return DPCLIP_ERR_UNSUPPORTED;    // candidate() checked dense rows
        if (!taken) return DPCLIP_ERR_INVALID_ARG;               // without `taken` the caller cannot know
        for (int i = 0; i < n; ++i) { done[idx[i]] = true; taken[idx[i]] = 1; }
    }
    if (clip_ld > 0) return DPCLIP_OK;
    for (int l0 = 0; l0 < L; ++l0) {
        if (done[l0] || !candidate(layers[l0])) continue;
        const dpclip_layer* grp[z::MAX_LAYERS];
        int idx[z::MAX_LAYERS];
        int n = 0;
        for (int l = l0; l < L && n < z::MAX_LAYERS; ++l) {
            const dpclip_layer& y = layers[l];
            if (done[l] || y.T != layers[l0].T || y.d_in != layers[l0].d_in || y.d_out != layers[l0].d_out) continue;
            if (!candidate(y) || (split && split[l] != split[l0])) continue;
            grp[n] = &y; idx[n] = l; ++n;
        }
        for (int i = 0; i < n; ++i) done[idx[i]] = true;
        if (n < 2) continue;
        {
            // Sharing a launch pays when a layer alone leaves every CTA a short row slice (pipeline fill and
            // epilogue then weigh heavily); layers that already give long slices keep their own launches,
            // whose one-wave split uses the SMs more evenly (measured on two 512 -> 2048 layers at
            // B*T = 32768: 174 us together on 128 CTAs, 2 x 80 us apart on 144).
            const dpclip_layer& y = layers[l0];
            const int bm = y.d_out > 128 && !(split && split[l0]) ? 256 : 128;
            const int tiles = ceil_div(y.d_out, bm) * ceil_div(y.d_in, z::BN);
            const long nkb = ceil_div((long)B * y.T, 64L);          // 64-row blocks
            const int ksplit = tiles < kNumSMs ? kNumSMs / tiles : 1;
            if (nkb / ksplit >= 32) continue;
        }
        const int rc = launch_zta_tc_group(grp, idx, n, B, clip, sigma * C, seed, stream_id0, workspace, workspace_bytes,
                                           (cudaStream_t)stream, split && split[l0]);
        if (rc < 0) return rc;
        if (rc == 0 && taken) for (int i = 0; i < n; ++i) taken[idx[i]] = 1;
        if (rc == 0 && !taken) return DPCLIP_ERR_INVALID_ARG;     // without `taken` the caller cannot know
    }
    return DPCLIP_OK;
}

int dpclip_factors(const float* sq_layers, int L, long ld_sq, int B, float C, float* clip, float* norms,
                   int* n_clipped, void* stream) {
    if (!sq_layers || !clip) return DPCLIP_ERR_INVALID_ARG;
    if (L <= 0 || B <= 0 || ld_sq < B || !(C > 0.f)) return DPCLIP_ERR_INVALID_ARG;
    factors_kernel<<<1, 256, 0, (cudaStream_t)stream>>>(sq_layers, L, ld_sq, B, C, clip, norms, n_clipped);
    return launch_status();
}

int dpclip_clipped_grad(const void* A, long lda, const void* Zbar, long ldz, int B, int T, int d_in,
                        int d_out, dpclip_dtype dtype, const float* clip, float* gW, long ldg, float* gb,
                        void* workspace, size_t workspace_bytes, void* stream) {
    int rc = check_layer_args(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype);
    if (rc) return rc;
    if (!gW || ldg < d_in) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(gW, 4) || (gb && !aligned_to(gb, 4))) return DPCLIP_ERR_MISALIGNED;
    if (!workspace || workspace_bytes < workspace_floor(B, T, d_in, d_out, dtype))
        return DPCLIP_ERR_WORKSPACE;
    return clipped_grad_impl(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype, clip, gW, ldg, gb, workspace,
                             workspace_bytes, nullptr, nullptr, (cudaStream_t)stream);
}

int dpclip_clipped_grad_noise(const void* A, long lda, const void* Zbar, long ldz, int B, int T, int d_in,
                              int d_out, dpclip_dtype dtype, const float* clip, float* gW, float* gb, float sigma,
                              float C, unsigned long long seed, unsigned long long stream_id_w,
                              unsigned long long stream_id_b, void* workspace, size_t workspace_bytes,
                              void* stream) {
    int rc = check_layer_args(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype);
    if (rc) return rc;
    if (!gW || !(sigma >= 0.f) || !(C >= 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(gW, 4) || (gb && !aligned_to(gb, 4))) return DPCLIP_ERR_MISALIGNED;
    if (!workspace || workspace_bytes < workspace_floor(B, T, d_in, d_out, dtype))
        return DPCLIP_ERR_WORKSPACE;
    NoiseSpec ns = {sigma * C, seed, stream_id_w, stream_id_b, true};
    bool noise_done = false;
    rc = clipped_grad_impl(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype, clip, gW, d_in, gb, workspace,
                           workspace_bytes, &ns, &noise_done, (cudaStream_t)stream);
    if (rc || noise_done) return rc;
    rc = dpclip_add_noise(gW, (size_t)d_out * d_in, sigma, C, seed, stream_id_w, stream);
    if (rc || !gb) return rc;
    return dpclip_add_noise(gb, (size_t)d_out, sigma, C, seed, stream_id_b, stream);
}

static int launch_dp_update(bool adam, float* theta, float* m, float* v, const float* gsum, size_t n, float inv_tau,
                            float C, float sigma, unsigned long long seed, unsigned long long stream_id, float lr,
                            float beta1, float beta2, float eps, int step, void* stream) {
    if (n == 0) return DPCLIP_OK;
    if (!theta || !gsum || (adam && (!m || !v))) return DPCLIP_ERR_INVALID_ARG;
    if (!(sigma >= 0.f) || !(C >= 0.f) || !(inv_tau > 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (adam && (step < 1 || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f))) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(theta, 4) || !aligned_to(gsum, 4) || (adam && (!aligned_to(m, 4) || !aligned_to(v, 4))))
        return DPCLIP_ERR_MISALIGNED;
    UpdateParams p;
    memset(&p, 0, sizeof(p));
    p.theta = theta; p.m = m; p.v = v; p.gsum = gsum; p.n = n;
    p.inv_tau = inv_tau; p.scale = sigma * C; p.lr = lr; p.beta1 = beta1; p.beta2 = beta2; p.eps = eps;
    if (adam) {
        p.inv_c1 = (float)(1.0 / (1.0 - pow((double)beta1, (double)step)));
        p.inv_c2 = (float)(1.0 / (1.0 - pow((double)beta2, (double)step)));
    }
    p.k0 = (uint32_t)seed; p.k1 = (uint32_t)(seed >> 32); p.s0 = (uint32_t)stream_id; p.s1 = (uint32_t)(stream_id >> 32);
    p.vec_ok = aligned_to(theta, 16) && aligned_to(gsum, 16) && (!adam || (aligned_to(m, 16) && aligned_to(v, 16)));
    const size_t nq = (n + 3) / 4;
    size_t blocks = (nq + 255) / 256;
    const size_t cap = (size_t)kNumSMs * 16;
    if (blocks > cap) blocks = cap;
    return launch_behind(adam ? dp_update_kernel<true> : dp_update_kernel<false>, dim3((unsigned)blocks), 256, 0, (cudaStream_t)stream, p);
}

int dpclip_dp_sgd_step(float* theta, const float* gsum, size_t n, float inv_tau, float C, float sigma,
                       unsigned long long seed, unsigned long long stream_id, float lr, void* stream) {
    return launch_dp_update(false, theta, nullptr, nullptr, gsum, n, inv_tau, C, sigma, seed, stream_id, lr, 0.f, 0.f,
                            0.f, 1, stream);
}

int dpclip_dp_adam_step(float* theta, float* m, float* v, const float* gsum, size_t n, float inv_tau, float C,
                        float sigma, unsigned long long seed, unsigned long long stream_id, float lr, float beta1,
                        float beta2, float eps, int step, void* stream) {
    return launch_dp_update(true, theta, m, v, gsum, n, inv_tau, C, sigma, seed, stream_id, lr, beta1, beta2, eps,
                            step, stream);
}

// Convolution layers given by their input feature map (implicit im2col).
static int conv_setup(SimtParams& p, const void* X, const void* Zbar, int z_channel_major, int B, const dpclip_conv* g,
                      int d_out, dpclip_dtype dtype, int has_bias, int* T_out) {
    if (!X || !Zbar || !g) return DPCLIP_ERR_INVALID_ARG;
    if (B <= 0 || d_out <= 0 || g->C <= 0 || g->H <= 0 || g->W <= 0 || g->kh <= 0 || g->kw <= 0 || g->stride <= 0 ||
        g->pad < 0) return DPCLIP_ERR_INVALID_ARG;
    if (dtype != DPCLIP_F32 && dtype != DPCLIP_BF16) return DPCLIP_ERR_INVALID_ARG;
    if (g->H + 2 * g->pad < g->kh || g->W + 2 * g->pad < g->kw) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(X, elt_size(dtype)) || !aligned_to(Zbar, elt_size(dtype))) return DPCLIP_ERR_MISALIGNED;
    const int Ho = (g->H + 2 * g->pad - g->kh) / g->stride + 1, Wo = (g->W + 2 * g->pad - g->kw) / g->stride + 1;
    const long T = (long)Ho * Wo, d_in = (long)g->C * g->kh * g->kw;
    if (T * B > 0x7FFFFFFFL || d_in > 0x7FFFFFFFL || (long)g->C * g->H * g->W > 0x7FFFFFFFL) return DPCLIP_ERR_INVALID_ARG;
    fill_simt_params(p, X, d_in, Zbar, d_out, (int)T, (int)d_in, d_out, has_bias, dtype);
    p.vec_a = 0;
    p.vec_z = z_channel_major ? 0 : vec4_ok(Zbar, d_out, dtype);
    p.cC = g->C; p.cH = g->H; p.cW = g->W; p.kh = g->kh; p.kw = g->kw; p.stride = g->stride; p.pad = g->pad;
    p.Wo = Wo; p.z_cm = z_channel_major ? 1 : 0;
    *T_out = (int)T;
    return DPCLIP_OK;
}

// fp32, dL/dZ as [B][T][d_out] with 16-byte rows, enough work: the tensor-core kernel with the A operand gathered
static bool conv_tf32_ok(const SimtParams& p, const void* X, const void* Zbar, int z_channel_major, int B, int T,
                         dpclip_dtype dtype, const void* workspace, size_t workspace_bytes, tc::ConvGather* cg) {
    if (path_switch(SW_FORCE_SIMT)) return false;
    if (dtype != DPCLIP_F32 || z_channel_major || !workspace || workspace_bytes < (size_t)kHeaderBytes) return false;
    if (!aligned_to(Zbar, 16) || p.d_out % 4 != 0 || p.kh > 255 || p.kw > 255) return false;
    if ((double)B * T * p.d_in * p.d_out < 32.0 * 1024 * 1024) return false;
    cg->X = static_cast<const float*>(X);
    cg->C = p.cC; cg->H = p.cH; cg->W = p.cW; cg->kh = p.kh; cg->kw = p.kw; cg->stride = p.stride; cg->pad = p.pad;
    cg->Wo = p.Wo;
    return true;
}

// bf16 convolution layers on the tensor cores (implicit im2col): see kernels_conv_tc.cuh for the restrictions
static bool conv_tc_ok(const SimtParams& p, const void* X, const void* Zbar, int z_channel_major, int B, int T,
                       dpclip_dtype dtype, const void* workspace, size_t workspace_bytes) {
    if (path_switch(SW_FORCE_SIMT)) return false;
    if (path_switch(SW_NO_CONV_TC)) return false;
    if (dtype != DPCLIP_BF16 || !workspace || workspace_bytes < (size_t)kHeaderBytes) return false;
    if (p.stride != 1 || !(p.Wo == 8 || p.Wo == 16 || p.Wo == 32 || p.Wo == 64) || T % 64 != 0) return false;
    if (p.d_out % 8 != 0 || p.d_out > 128) return false;
    const long x_elems = (long)p.cC * p.cH * p.cW;
    if (x_elems * 2 > tc::ctc::X_BYTES || x_elems % 8 != 0) return false;
    return aligned_to(X, 16) && aligned_to(Zbar, 16);
}

extern "C++" {
template <bool GRAD>
static int launch_conv_tc(const SimtParams& sp, const void* X, const void* Zbar, int B, int T, int has_bias,
                          const float* clip, float* sq, float* gW, long ldg, float* gb, void* workspace,
                          size_t workspace_bytes, cudaStream_t st, const NoiseSpec* noise = nullptr, bool* noise_done = nullptr) {
    namespace c = tc::ctc;
    CUtensorMap mz;
    // dL/dZ as [B][T][d_out]: boxes of 64 rows t x 64 columns; as [B][d_out][T]: one box of d_out rows x 64 t
    if (sp.z_cm ? !make_map_bf16(&mz, Zbar, (long)B * sp.d_out, T, T, c::BK, sp.d_out)
                : !make_map_bf16(&mz, Zbar, (long)B * T, sp.d_out, sp.d_out, 64, c::BK)) return DPCLIP_ERR_CUDA;
    c::Params p;
    memset(&p, 0, sizeof(p));
    p.z_cm = sp.z_cm;
    p.X = static_cast<const __nv_bfloat16*>(X);
    p.B = B; p.C = sp.cC; p.H = sp.cH; p.W = sp.cW; p.kh = sp.kh; p.kw = sp.kw; p.pad = sp.pad;
    p.Wo = sp.Wo; p.Ho = T / sp.Wo;
    p.wo_shift = sp.Wo == 8 ? 3 : sp.Wo == 16 ? 4 : sp.Wo == 32 ? 5 : 6;
    p.T = T; p.d_in = sp.d_in; p.d_out = sp.d_out; p.has_bias = has_bias ? 1 : 0;
    p.tiles_n = ceil_div(sp.d_in + p.has_bias, c::BN);
    p.status = static_cast<int*>(workspace);
    int slices = 1;
    if (GRAD) {
        // one wave: as many slices of examples as there are SMs per block of patch columns
        slices = sm_budget() / p.tiles_n;
        if (slices > B) slices = B;
        if (slices < 1) slices = 1;
        p.ex_per_item = ceil_div(B, slices);
        slices = ceil_div(B, p.ex_per_item);
        p.n_items = slices * p.tiles_n;
        const size_t part_bytes = (size_t)p.n_items * 128 * c::BN * 4;
        if (workspace_bytes < (size_t)kHeaderBytes + part_bytes) return 1;        // the caller takes the fp32-ALU kernel
        p.part = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes);
        p.clip = clip;
    } else {
        p.ex_per_item = 1;
        p.n_items = B * p.tiles_n;
        p.sq = sq;
        if (!clear_sq(sq, (size_t)B, st)) return DPCLIP_ERR_CUDA;
    }
    if (!enable_smem(tc::conv_tc_kernel<GRAD>, c::SMEM_BYTES)) return DPCLIP_ERR_CUDA;
    const int grid = p.n_items < sm_budget() ? p.n_items : sm_budget();
    tc::conv_tc_kernel<GRAD><<<grid, c::THREADS, c::SMEM_BYTES, st>>>(mz, p);
    int rc = launch_status();
    if (rc || !GRAD) return rc;
    // fixed-order sum of the slices' tiles; the bias sums are column d_in of the tiles
    tc::zta::Params zp;
    memset(&zp, 0, sizeof(zp));
    zp.part = p.part; zp.tiles_n = p.tiles_n; zp.vec_ok = aligned_to(gW, 16) && ldg % 4 == 0;
    tc::ReduceParams r;
    memset(&r, 0, sizeof(r));
    r.part = p.part; r.n_tiles = p.tiles_n; r.tiles_n = p.tiles_n; r.ksplit = slices; r.BM = 128; r.BN = c::BN;
    r.d_out = sp.d_out; r.d_in = sp.d_in; r.gW = gW; r.ldg = ldg; r.gb = gb; r.vec_ok = zp.vec_ok;
    r.bias_col = 1;
    if (noise && noise->scale > 0.f && ldg == sp.d_in) {
        r.noise_scale = noise->scale;
        r.k0 = (uint32_t)noise->seed; r.k1 = (uint32_t)(noise->seed >> 32);
        r.sw0 = (uint32_t)noise->sid_w; r.sw1 = (uint32_t)(noise->sid_w >> 32);
        r.sb0 = (uint32_t)noise->sid_b; r.sb1 = (uint32_t)(noise->sid_b >> 32);
        if (noise_done) *noise_done = true;
    }
    const long n_vec = (long)sp.d_out * ((sp.d_in + 3) / 4);
    int lanes = 1;
    while (lanes < 8 && lanes * 2 <= slices && n_vec * lanes < 2L * kNumSMs * 256) lanes *= 2;
    r.lanes = lanes;
    long blocks = (n_vec + (256 / lanes) - 1) / (256 / lanes);
    if (blocks > 8L * kNumSMs) blocks = 8L * kNumSMs;
    return launch_behind(tc::reduce_partials_kernel, dim3((unsigned)blocks), 256, 0, st, r);
}
}  // extern "C++"

// fp32 dL/dZ in the channel-major layout [B][d_out][T]: the tf32 tensor-core kernel reads [row][feature]
// tiles, so the tensor is rewritten once per call as [B][T][d_out] behind the partial-tile scratch when the
// workspace has room for it (dpclip_conv_workspace_bytes); otherwise the fp32-ALU kernel reads it in place.
// Returns the pointer to use and clears *channel_major when it did.
static const void* conv_f32_rows_of_channel_major(const SimtParams& p, const void* Zbar, int* channel_major, int B, int T,
                                                  dpclip_dtype dtype, void* workspace, size_t workspace_bytes,
                                                  cudaStream_t st, int* rc) {
    *rc = DPCLIP_OK;
    if (dtype != DPCLIP_F32 || !*channel_major || !workspace || B > 65535) return Zbar;
    if (path_switch(SW_FORCE_SIMT)) return Zbar;
    if (p.d_out % 4 != 0 || p.kh > 255 || p.kw > 255) return Zbar;
    if ((double)B * T * p.d_in * p.d_out < 32.0 * 1024 * 1024) return Zbar;           // stays on the fp32-ALU tiles
    const size_t z_bytes = (size_t)B * T * p.d_out * 4;
    if (workspace_bytes < (size_t)kHeaderBytes + kTcScratchBytes + z_bytes) return Zbar;
    float* rows = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes + kTcScratchBytes);
    const dim3 grid(ceil_div(T, 32), ceil_div(p.d_out, 32), B);
    channel_major_to_rows_kernel<<<grid, 256, 0, st>>>(static_cast<const float*>(Zbar), rows, p.d_out, T);
    if (launch_status()) { *rc = DPCLIP_ERR_CUDA; return Zbar; }
    *channel_major = 0;
    return rows;
}

// fp32 first layers with at most 32 patch columns and 32 outputs: write the patch matrix out behind the scratch
// areas above and hand it to the dense entry points (packed narrow tensor-core kernel).  Needs dL/dZ as rows.
// Returns the patch matrix, or NULL when the layer does not qualify or the workspace has no room.
static const float* conv_f32_narrow_patches(const SimtParams& p, const void* X, const void* z_rows, int z_cm, int B, int T,
                                            dpclip_dtype dtype, int has_bias, void* workspace, size_t workspace_bytes,
                                            cudaStream_t st, int* rc) {
    *rc = DPCLIP_OK;
    if (dtype != DPCLIP_F32 || z_cm || !workspace || p.d_out > 32 || p.d_in + (has_bias ? 1 : 0) > 32) return nullptr;
    if (path_switch(SW_FORCE_SIMT)) return nullptr;
    if (path_switch(SW_NO_CONV_PATCHES)) return nullptr;
    if ((double)B * T * p.d_in * p.d_out < 32.0 * 1024 * 1024) return nullptr;
    if (((long)T * p.d_in * 4) % 16 != 0 || ((long)T * p.d_out * 4) % 16 != 0 || !aligned_to(z_rows, 16)) return nullptr;
    const size_t z_bytes = round_up((size_t)B * T * p.d_out * 4, 256), a_bytes = (size_t)B * T * p.d_in * 4;
    if (workspace_bytes < (size_t)kHeaderBytes + kTcScratchBytes + z_bytes + a_bytes) return nullptr;
    float* patches = reinterpret_cast<float*>(static_cast<char*>(workspace) + kHeaderBytes + kTcScratchBytes + z_bytes);
    const long rows = (long)B * T;
    if (rows > 0x7FFFFFFFL - 64) return nullptr;
    im2col_f32_kernel<<<(unsigned)((rows + 63) / 64), 256, 0, st>>>(static_cast<const float*>(X), patches, (int)rows, T,
                                                                    p.d_in, p.cC, p.cH, p.cW, p.kh, p.kw, p.stride, p.pad,
                                                                    p.Wo);
    if (launch_status()) { *rc = DPCLIP_ERR_CUDA; return nullptr; }
    return patches;
}

size_t dpclip_conv_workspace_bytes(int B, const dpclip_conv* geom, int d_out, dpclip_dtype dtype, int z_channel_major) {
    if (!geom || B <= 0 || d_out <= 0 || geom->stride <= 0) return kHeaderBytes;
    const int Ho = (geom->H + 2 * geom->pad - geom->kh) / geom->stride + 1;
    const int Wo = (geom->W + 2 * geom->pad - geom->kw) / geom->stride + 1;
    if (Ho <= 0 || Wo <= 0) return kHeaderBytes;
    const int T = Ho * Wo;
    size_t w = dpclip_workspace_bytes(B, T, geom->C * geom->kh * geom->kw, d_out, dtype, DPCLIP_AUTO);
    if (dtype == DPCLIP_F32 && w >= (size_t)kHeaderBytes + kTcScratchBytes) {
        const int d_in = geom->C * geom->kh * geom->kw;
        const bool narrow = d_out <= 32 && d_in + 1 <= 32;
        if (z_channel_major || narrow) w += round_up((size_t)B * T * d_out * 4, 256);   // the row-major copy of dL/dZ
        if (narrow) w += (size_t)B * T * d_in * 4;                                       // the patch matrix
    }
    return w;
}

int dpclip_conv_sqnorms(const void* X, const void* Zbar, int z_channel_major, int B, const dpclip_conv* geom,
                        int d_out, dpclip_dtype dtype, int has_bias, float* sq_layer, void* workspace,
                        size_t workspace_bytes, void* stream) {
    SimtParams p;
    int T = 0;
    int rc = conv_setup(p, X, Zbar, z_channel_major, B, geom, d_out, dtype, has_bias, &T);
    if (rc) return rc;
    if (!sq_layer) return DPCLIP_ERR_INVALID_ARG;
    if (B > 65535) return DPCLIP_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    tc::ConvGather cg;
    if (conv_tc_ok(p, X, Zbar, z_channel_major, B, T, dtype, workspace, workspace_bytes))
        return launch_conv_tc<false>(p, X, Zbar, B, T, has_bias, nullptr, sq_layer, nullptr, 0, nullptr, workspace,
                                     workspace_bytes, st);
    int z_cm = z_channel_major;
    const void* z_rows = conv_f32_rows_of_channel_major(p, Zbar, &z_cm, B, T, dtype, workspace, workspace_bytes, st, &rc);
    if (rc) return rc;
    if (const float* patches = conv_f32_narrow_patches(p, X, z_rows, z_cm, B, T, dtype, has_bias, workspace, workspace_bytes,
                                                       st, &rc))
        return dpclip_layer_sqnorms(patches, p.d_in, z_rows, d_out, B, T, p.d_in, d_out, dtype, has_bias, DPCLIP_AUTO,
                                    sq_layer, workspace, (size_t)kHeaderBytes + kTcScratchBytes, stream);
    if (rc) return rc;
    if (conv_tf32_ok(p, X, z_rows, z_cm, B, T, dtype, workspace, workspace_bytes, &cg))
        return launch_zta_tf32(nullptr, p.d_in, z_rows, d_out, B, T, p.d_in, d_out, true, has_bias, nullptr, nullptr, 0,
                               nullptr, sq_layer, workspace, workspace_bytes, nullptr, nullptr, st, &cg);
    const int n_tiles = p.tiles_m * p.tiles_n;
    int split = ceil_div(2 * kNumSMs, B);
    if (split > n_tiles) split = n_tiles;
    if (split < 1) split = 1;
    p.sq = sq_layer;
    p.use_atomic = split > 1;
    if (p.use_atomic && !clear_sq(sq_layer, (size_t)B, st)) return DPCLIP_ERR_CUDA;
    dim3 grid(split, B);
    if (dtype == DPCLIP_F32) zta_simt_kernel<float, false, true><<<grid, SIMT_THREADS, 0, st>>>(p);
    else zta_simt_kernel<__nv_bfloat16, false, true><<<grid, SIMT_THREADS, 0, st>>>(p);
    return launch_status();
}

static int conv_clipped_grad_impl(const void* X, const void* Zbar, int z_channel_major, int B, const dpclip_conv* geom,
                                  int d_out, dpclip_dtype dtype, const float* clip, float* gW, long ldg, float* gb,
                                  void* workspace, size_t workspace_bytes, const NoiseSpec* noise, bool* noise_done,
                                  void* stream) {
    SimtParams p;
    int T = 0;
    int rc = conv_setup(p, X, Zbar, z_channel_major, B, geom, d_out, dtype, gb != nullptr, &T);
    if (rc) return rc;
    if (!gW || ldg < p.d_in) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(gW, 4) || (gb && !aligned_to(gb, 4))) return DPCLIP_ERR_MISALIGNED;
    cudaStream_t st = (cudaStream_t)stream;
    tc::ConvGather cg;
    if (conv_tc_ok(p, X, Zbar, z_channel_major, B, T, dtype, workspace, workspace_bytes)) {
        rc = launch_conv_tc<true>(p, X, Zbar, B, T, gb != nullptr, clip, nullptr, gW, ldg, gb, workspace, workspace_bytes, st, noise,
                                  noise_done);
        if (rc <= 0) return rc;
    }
    int z_cm = z_channel_major;
    const void* z_rows = conv_f32_rows_of_channel_major(p, Zbar, &z_cm, B, T, dtype, workspace, workspace_bytes, st, &rc);
    if (rc) return rc;
    if (const float* patches = conv_f32_narrow_patches(p, X, z_rows, z_cm, B, T, dtype, gb != nullptr, workspace,
                                                       workspace_bytes, st, &rc))
        return clipped_grad_impl(patches, p.d_in, z_rows, d_out, B, T, p.d_in, d_out, dtype, clip, gW, ldg, gb, workspace,
                                 (size_t)kHeaderBytes + kTcScratchBytes, noise, noise_done, st);
    if (rc) return rc;
    if (conv_tf32_ok(p, X, z_rows, z_cm, B, T, dtype, workspace, workspace_bytes, &cg) &&
        workspace_bytes >= (size_t)kHeaderBytes + kTcScratchBytes)
        return launch_zta_tf32(nullptr, p.d_in, z_rows, d_out, B, T, p.d_in, d_out, false, 0, clip, gW, ldg, gb, nullptr,
                               workspace, workspace_bytes, noise, noise_done, st, &cg);
    const int n_tiles = p.tiles_m * p.tiles_n;
    const long rows = (long)B * T;
    long ksplit = ceil_div(4 * kNumSMs, n_tiles);
    const long max_split = (rows + 4 * SIMT_BK - 1) / (4 * SIMT_BK);
    if (ksplit > max_split) ksplit = max_split;
    if (ksplit < 1) ksplit = 1;
    if (ksplit > 65535) ksplit = 65535;
    long per = (rows + ksplit - 1) / ksplit;
    per = (per + SIMT_BK - 1) / SIMT_BK * SIMT_BK;
    ksplit = (rows + per - 1) / per;
    p.clip = clip; p.gW = gW; p.ldg = ldg; p.gb = gb;
    p.rows_total = rows; p.rows_per_split = per;
    p.use_atomic = ksplit > 1;
    if (p.use_atomic) {
        if (cudaMemset2DAsync(gW, sizeof(float) * (size_t)ldg, 0, sizeof(float) * (size_t)p.d_in, d_out, st) != cudaSuccess)
            return DPCLIP_ERR_CUDA;
        if (gb && cudaMemsetAsync(gb, 0, sizeof(float) * (size_t)d_out, st) != cudaSuccess) return DPCLIP_ERR_CUDA;
    }
    simt_noise(p, noise, noise_done);
    dim3 grid(n_tiles, (unsigned)ksplit);
    if (dtype == DPCLIP_F32) zta_simt_kernel<float, true, true><<<grid, SIMT_THREADS, 0, st>>>(p);
    else zta_simt_kernel<__nv_bfloat16, true, true><<<grid, SIMT_THREADS, 0, st>>>(p);
    return launch_status();
}

int dpclip_conv_clipped_grad(const void* X, const void* Zbar, int z_channel_major, int B, const dpclip_conv* geom,
                             int d_out, dpclip_dtype dtype, const float* clip, float* gW, long ldg, float* gb,
                             void* workspace, size_t workspace_bytes, void* stream) {
    return conv_clipped_grad_impl(X, Zbar, z_channel_major, B, geom, d_out, dtype, clip, gW, ldg, gb, workspace, workspace_bytes,
                                  nullptr, nullptr, stream);
}

int dpclip_step_noise(const dpclip_layer* layers, int L, float C, float sigma, unsigned long long seed,
                      unsigned long long stream_id0, void* stream) {
    if (!layers || L <= 0 || !(C >= 0.f) || !(sigma >= 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (sigma * C == 0.f) return DPCLIP_OK;
    cudaStream_t st = (cudaStream_t)stream;
    for (int l0 = 0; l0 < L; l0 += NOISE_BATCH_MAX / 2) {          // at most 64 layers (128 tensors) per launch
        NoiseBatchParams p;
        memset(&p, 0, sizeof(p));
        p.scale = sigma * C; p.k0 = (uint32_t)seed; p.k1 = (uint32_t)(seed >> 32);
        int blocks = 0;
        const int l1 = l0 + NOISE_BATCH_MAX / 2 < L ? l0 + NOISE_BATCH_MAX / 2 : L;
        for (int l = l0; l < l1; ++l) {
            const dpclip_layer& y = layers[l];
            if (!y.gW || y.d_in <= 0 || y.d_out <= 0) return DPCLIP_ERR_INVALID_ARG;
            if (y.ldg != y.d_in) return DPCLIP_ERR_UNSUPPORTED;      // noise indexes the dense tensor
            if (y.has_bias && !y.gb) return DPCLIP_ERR_INVALID_ARG;
            if (!aligned_to(y.gW, 4) || (y.gb && !aligned_to(y.gb, 4))) return DPCLIP_ERR_MISALIGNED;
            auto add = [&](float* g, size_t n, unsigned long long sid) {
                const size_t nq = (n + 3) / 4;
                size_t b = (nq + 255) / 256;
                if (b > (size_t)kNumSMs * 4) b = (size_t)kNumSMs * 4;
                p.g[p.count] = g; p.n[p.count] = n; p.sid[p.count] = sid; p.blk_begin[p.count] = blocks;
                blocks += (int)b; ++p.count;
            };
            add(y.gW, (size_t)y.d_out * y.d_in, stream_id0 + 2ull * l);
            if (y.has_bias) add(y.gb, (size_t)y.d_out, stream_id0 + 2ull * l + 1);
        }
        p.blk_begin[p.count] = blocks;
        noise_batch_kernel<<<blocks, 256, 0, st>>>(p);
        if (launch_status()) return DPCLIP_ERR_CUDA;
    }
    return DPCLIP_OK;
}

int dpclip_t1_layers_supported(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype) {
    if (!layers || L <= 0 || B <= 0) return 0;
    T1Group g;
    if (prepare_t1_group(g, layers, L, B, dtype, 1.f, 0.f, 0, 0, nullptr, nullptr, /*mixed_only=*/false)) return 0;
    return g.active ? 1 : 0;
}

int dpclip_t1_layers_sqnorms(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float* sq_layers,
                             void* stream) {
    if (!layers || L <= 0 || B <= 0 || !sq_layers) return DPCLIP_ERR_INVALID_ARG;
    T1Group g;
    int rc = prepare_t1_group(g, layers, L, B, dtype, 1.f, 0.f, 0, 0, sq_layers, nullptr, /*mixed_only=*/false);
    if (rc) return rc;
    if (!g.active) return DPCLIP_ERR_UNSUPPORTED;
    if (dtype == DPCLIP_F32) t1_all_norms_kernel<float><<<g.p.L * B, 128, 0, (cudaStream_t)stream>>>(g.p);
    else t1_all_norms_kernel<__nv_bfloat16><<<g.p.L * B, 128, 0, (cudaStream_t)stream>>>(g.p);
    return launch_status();
}

int dpclip_t1_layers_clipped_grad_noise(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype,
                                        const float* clip, float C, float sigma, unsigned long long seed,
                                        unsigned long long stream_id0, void* workspace, size_t workspace_bytes,
                                        void* stream) {
    if (!layers || L <= 0 || B <= 0 || !clip) return DPCLIP_ERR_INVALID_ARG;
    if (!(C > 0.f) || !(sigma >= 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < (size_t)kHeaderBytes) return DPCLIP_ERR_WORKSPACE;
    T1Group g;
    int rc = prepare_t1_group(g, layers, L, B, dtype, C, sigma, seed, stream_id0, nullptr, clip, /*mixed_only=*/false);
    if (rc) return rc;
    if (!g.active) return DPCLIP_ERR_UNSUPPORTED;
    rc = launch_fused_t1_tf32(g.p, false, dtype, workspace, workspace_bytes, (cudaStream_t)stream);
    return rc > 0 ? DPCLIP_ERR_UNSUPPORTED : rc;
}

// per_example: [B][2][d] for the examples' gradients (scale, shift), or NULL
static int elementwise_sqnorms(const void* Hbar, long ldh, const void* Zbar, long ldz, int B, int T, int d, dpclip_dtype dtype,
                               int has_shift, float* sq_layer, float* per_example, void* stream) {
    int rc = check_layer_args(Hbar, ldh, Zbar, ldz, B, T, d, d, dtype);
    if (rc) return rc;
    if (!sq_layer) return DPCLIP_ERR_INVALID_ARG;
    if (B > 65535) return DPCLIP_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    const bool vec = vec4_ok(Hbar, ldh, dtype) && vec4_ok(Zbar, ldz, dtype) && d % 4 == 0;
    const int v = vec ? 4 : 1;
    const int cg = (long)ceil_div(d, 64 * v) * B >= 4L * kNumSMs ? 64 : 32;
    const dim3 grid(ceil_div(d, cg * v), B);
    const int use_atomic = grid.x > 1;
    if (use_atomic && !clear_sq(sq_layer, (size_t)B, st)) return DPCLIP_ERR_CUDA;
    if (dtype == DPCLIP_F32) launch_ew_norm<float>(vec, cg, grid, st, Hbar, ldh, Zbar, ldz, T, d, has_shift, sq_layer, use_atomic, per_example);
    else launch_ew_norm<__nv_bfloat16>(vec, cg, grid, st, Hbar, ldh, Zbar, ldz, T, d, has_shift, sq_layer, use_atomic, per_example);
    return launch_status();
}
int dpclip_elementwise_sqnorms(const void* Hbar, long ldh, const void* Zbar, long ldz, int B, int T, int d,
                               dpclip_dtype dtype, int has_shift, float* sq_layer, void* stream) {
    return elementwise_sqnorms(Hbar, ldh, Zbar, ldz, B, T, d, dtype, has_shift, sq_layer, nullptr, stream);
}

int dpclip_elementwise_clipped_grad(const void* Hbar, long ldh, const void* Zbar, long ldz, int B, int T, int d,
                                    dpclip_dtype dtype, const float* clip, float* g_scale, float* g_shift,
                                    void* stream) {
    int rc = check_layer_args(Hbar, ldh, Zbar, ldz, B, T, d, d, dtype);
    if (rc) return rc;
    if (!g_scale) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(g_scale, 4) || (g_shift && !aligned_to(g_shift, 4))) return DPCLIP_ERR_MISALIGNED;
    cudaStream_t st = (cudaStream_t)stream;
    const bool vec = vec4_ok(Hbar, ldh, dtype) && vec4_ok(Zbar, ldz, dtype) && d % 4 == 0;
    const int v = vec ? 4 : 1;
    const long R = (long)B * T;
    const int cg = 64;
    const int col_blocks = ceil_div(d, cg * v);
    // about eight CTAs per SM in all (measured: 190 vs 217 us with four on 1 GB of bf16 input), and at least
    // 256 rows per CTA: every CTA ends with one atomic per column, and with 64-row CTAs those adds (512 per
    // address at B*T = 32768, d = 512) cost more than the rows (38.9 vs 26.6 us)
    long slices = (8L * kNumSMs + col_blocks - 1) / col_blocks;
    if (slices > (R + 255) / 256) slices = (R + 255) / 256;
    if (slices < 1) slices = 1;
    if (slices > 65535) slices = 65535;
    const long rows_per_cta = (R + slices - 1) / slices;
    const dim3 grid(col_blocks, (unsigned)ceil_div(R, rows_per_cta));
    if (cudaMemsetAsync(g_scale, 0, sizeof(float) * (size_t)d, st) != cudaSuccess) return DPCLIP_ERR_CUDA;
    if (g_shift && cudaMemsetAsync(g_shift, 0, sizeof(float) * (size_t)d, st) != cudaSuccess) return DPCLIP_ERR_CUDA;
    if (dtype == DPCLIP_F32) launch_ew_grad<float>(vec, cg, grid, st, Hbar, ldh, Zbar, ldz, R, rows_per_cta, T, d, clip, g_scale, g_shift);
    else launch_ew_grad<__nv_bfloat16>(vec, cg, grid, st, Hbar, ldh, Zbar, ldz, R, rows_per_cta, T, d, clip, g_scale, g_shift);
    return launch_status();
}

int dpclip_add_noise(float* g, size_t n, float sigma, float C, unsigned long long seed,
                     unsigned long long stream_id, void* stream) {
    if (n == 0) return DPCLIP_OK;
    if (!g || !(sigma >= 0.f) || !(C >= 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(g, 4)) return DPCLIP_ERR_MISALIGNED;
    if (sigma * C == 0.f) return DPCLIP_OK;          // nothing to add: no launch
    const size_t nq = (n + 3) / 4;
    size_t blocks = (nq + 255) / 256;
    const size_t cap = (size_t)kNumSMs * 16;
    if (blocks > cap) blocks = cap;
    noise_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(
        g, n, sigma * C, (uint32_t)seed, (uint32_t)(seed >> 32), (uint32_t)stream_id,
        (uint32_t)(stream_id >> 32), aligned_to(g, 16) ? 1 : 0);
    return launch_status();
}

// Norms / clipped sum + noise of a layer that is not a dense product (element-wise parameters, convolution
// given by its feature map): the per-layer entry points, with the layer's row of sq and its noise streams.
static int other_kind_sqnorms(const dpclip_model_layer& m, int B, dpclip_dtype dtype, float* sq_row, float* per_example,
                              void* workspace, size_t workspace_bytes, void* stream) {
    const dpclip_layer& y = m.layer;
    if (m.kind == DPCLIP_KIND_ELEMENTWISE) {
        if (y.d_in != y.d_out) return DPCLIP_ERR_INVALID_ARG;
        return elementwise_sqnorms(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, dtype, y.has_bias, sq_row, per_example, stream);
    }
    if (m.kind == DPCLIP_KIND_CONV)
        return dpclip_conv_sqnorms(y.A, y.Zbar, m.z_channel_major, B, &m.conv, y.d_out, dtype, y.has_bias, sq_row,
                                   workspace, workspace_bytes, stream);
    return DPCLIP_ERR_INVALID_ARG;
}

static int other_kind_clipped_grad_noise(const dpclip_model_layer& m, int B, dpclip_dtype dtype, const float* clip,
                                         float C, float sigma, unsigned long long seed, unsigned long long sid_w,
                                         unsigned long long sid_b, void* workspace, size_t workspace_bytes,
                                         void* stream) {
    const dpclip_layer& y = m.layer;
    float* gb = y.has_bias ? y.gb : nullptr;
    if (!y.gW || (y.has_bias && !gb)) return DPCLIP_ERR_INVALID_ARG;
    size_t n_w = 0;
    int rc;
    if (m.kind == DPCLIP_KIND_ELEMENTWISE) {
        if (y.d_in != y.d_out) return DPCLIP_ERR_INVALID_ARG;
        rc = dpclip_elementwise_clipped_grad(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, dtype, clip, y.gW, gb, stream);
        n_w = (size_t)y.d_in;
    } else if (m.kind == DPCLIP_KIND_CONV) {
        const long d_in = (long)m.conv.C * m.conv.kh * m.conv.kw;
        if (y.ldg != d_in) return DPCLIP_ERR_UNSUPPORTED;        // noise indexes the dense tensor
        const NoiseSpec ns = {sigma * C, seed, sid_w, sid_b};
        bool noise_done = false;
        rc = conv_clipped_grad_impl(y.A, y.Zbar, m.z_channel_major, B, &m.conv, y.d_out, dtype, clip, y.gW, y.ldg, gb,
                                    workspace, workspace_bytes, &ns, &noise_done, stream);
        if (rc || noise_done) return rc;
        n_w = (size_t)y.d_out * (size_t)d_in;
    } else {
        return DPCLIP_ERR_INVALID_ARG;
    }
    if (rc) return rc;
    rc = dpclip_add_noise(y.gW, n_w, sigma, C, seed, sid_w, stream);
    if (rc) return rc;
    if (gb) rc = dpclip_add_noise(gb, m.kind == DPCLIP_KIND_ELEMENTWISE ? (size_t)y.d_in : (size_t)y.d_out, sigma, C,
                                  seed, sid_b, stream);
    return rc;
}

// Per-example gradients of element-wise layers between the two stages of a step ([B][2][d] per layer).  Layers of fewer than 8
// positions keep their second pass: their inputs are about as many bytes.
static size_t ew_rows_bytes(const dpclip_model_layer& m, int B) {
    const dpclip_layer& y = m.layer;
    if (m.kind != DPCLIP_KIND_ELEMENTWISE || y.T < 8 || y.d_in <= 0 || y.d_in != y.d_out || B <= 0) return 0;
    return round_up((size_t)B * 2 * y.d_in * sizeof(float), 256);
}
static size_t ew_rows_total(const dpclip_model_layer* layers, int L, int B) {
    size_t total = 0;
    for (int l = 0; l < L; ++l) total += ew_rows_bytes(layers[l], B);
    return total;
}
// Clipped sums with noise of the element-wise layers whose per-example gradients are there.
static int ew_rows_grads(const dpclip_model_layer* other, float* const* rows, int L, int B, const float* clip, float C, float sigma,
                         unsigned long long seed, unsigned long long stream_id0, cudaStream_t st) {
    EwRowsParams p;
    int blocks = 0;
    p.n = 0; p.B = B; p.clip = clip; p.noise_scale = sigma * C; p.k0 = (uint32_t)seed; p.k1 = (uint32_t)(seed >> 32);
    p.cluster = 1;
    while (p.cluster < EW_ROWS_MAX_CLUSTER && (long)p.cluster * EW_ROWS_PER_CTA < B) p.cluster *= 2;
    for (int l = 0; l < L; ++l) {
        if (rows[l]) {
            const dpclip_layer& y = other[l].layer;
            const unsigned long long sw = stream_id0 + 2ull * l, sb = sw + 1;
            EwRowsLayer& q = p.layer[p.n++];
            q.rows = rows[l]; q.g_scale = y.gW; q.g_shift = y.has_bias ? y.gb : nullptr; q.d = y.d_in; q.blk_begin = blocks;
            q.sw0 = (uint32_t)sw; q.sw1 = (uint32_t)(sw >> 32); q.sb0 = (uint32_t)sb; q.sb1 = (uint32_t)(sb >> 32);
            blocks += ceil_div(y.d_in, 32L) * (q.g_shift ? 2 : 1);
        }
        if (p.n == EW_ROWS_MAX_LAYERS || (l == L - 1 && p.n > 0)) {
            if (B <= EW_ROWS_FEW) elementwise_rows_grad_kernel<EW_THREADS / 32, false><<<blocks, EW_THREADS, 0, st>>>(p);
            else if (p.cluster == 1) elementwise_rows_grad_kernel<EW_ROWS_WARPS, false><<<blocks, 32 * EW_ROWS_WARPS, 0, st>>>(p);
            else {
                cudaLaunchConfig_t cfg;
                memset(&cfg, 0, sizeof(cfg));
                cfg.gridDim = dim3(blocks * p.cluster); cfg.blockDim = dim3(32 * EW_ROWS_WARPS); cfg.stream = st;
                cudaLaunchAttribute attr;
                attr.id = cudaLaunchAttributeClusterDimension;
                attr.val.clusterDim.x = p.cluster; attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
                cfg.attrs = &attr; cfg.numAttrs = 1;
                if (cudaLaunchKernelEx(&cfg, elementwise_rows_grad_kernel<EW_ROWS_WARPS, true>, p) != cudaSuccess) { cudaGetLastError(); return DPCLIP_ERR_CUDA; }
            }
            if (launch_status()) return DPCLIP_ERR_CUDA;
            p.n = 0; blocks = 0;
        }
    }
    return DPCLIP_OK;
}

// ---------------------------------------------------------------------------
// Operand staging of a whole step (kernels_stage.cuh): which layers' operands are rewritten, where the copies lie, and
// the layers as the rest of the step sees them.  The copies lie behind the scratch, in lane 0's workspace, and live
// from the first launch of the step to its last.
// ---------------------------------------------------------------------------
constexpr int kStageMaxLayers = 64;
constexpr int kLongRow = 64;
// Copies of one step; a layer that no longer fits keeps its fp32-ALU form.
constexpr size_t kStageCapBytes = (size_t)3 << 30;
struct StagePlan {
    bool active = false;
    dpclip_layer eff[kStageMaxLayers];       // T = 0: a layer of another kind
    bool other[kStageMaxLayers];             // goes through the entry points of its kind (not staged, not dense)
    bool split[kStageMaxLayers];             // clipped sum with two-term scaled operands (see zta_tc_kernel)
    dpclip_dtype t1_dtype;                   // type of the T = 1 layers after staging
    stage::Job job[2 * kStageMaxLayers];
    int n_jobs = 0, smem = 0;
    size_t scratch = 0, bytes = 0;           // bytes before the copies, and with them
};

// Copying pays once a layer (T > 1) has real contraction work: below 2^25 multiply-adds the fp32-ALU kernels take about as
// long as the copy's own launch (66 -> 66 features at B = 64, T = 32: 34 us a step either way; 130 -> 130 there, 35 M:
// 35.1 staged, 41.1 not; 250 -> 250 at T = 128, 512 M: 37 / 119 us).  With few rows the tensor-core kernels fill few SMs: 501
// -> 501 at B*T = 256 (64 M) 47 / 40 us, 1001 -> 1001 there 53 / 82 us.
static bool stage_worth_it(double rows, double weights, dpclip_dtype dtype) {
    const double macs = rows * weights;
    return macs >= 32.0 * 1024 * 1024 && (dtype == DPCLIP_F32 || rows >= 1024 || macs >= 128e6);
}

static bool stage_plan(StagePlan& sp, const dpclip_layer* layers, const dpclip_model_layer* other, int L, int B,
                       dpclip_dtype dtype, char* base, bool t1_too) {
    sp.active = false;
    if (L > kStageMaxLayers || path_switch(SW_FORCE_SIMT) || path_switch(SW_NO_STAGE)) return false;
    const size_t es = elt_size(dtype);
    const int unit = 16 / (int)es;                                  // elements of 16 bytes
    sp.n_jobs = 0; sp.smem = 0; sp.t1_dtype = dtype;
    size_t off = 0;                                                 // within the area of copies
    bool any = false;
    struct Take { int job; size_t off; int layer; bool z; };
    Take takes[2 * kStageMaxLayers];
    auto add_job = [&](int l, bool z, int kind, const void* src, long src_ld, int dst_ld, int rows, int cols, size_t dst_es) -> stage::Job& {
        stage::Job& j = sp.job[sp.n_jobs];
        memset(&j, 0, sizeof(j));
        j.kind = kind; j.es = (int)es; j.src = src; j.src_ld = src_ld; j.dst_ld = dst_ld; j.rows = rows; j.cols = cols;
        takes[sp.n_jobs] = {sp.n_jobs, off, l, z};
        off += round_up((size_t)rows * dst_ld * dst_es, 256);
        ++sp.n_jobs;
        return j;
    };
    auto misaligned = [&](const void* ptr, long ld) { return !aligned_to(ptr, 16) || ld % unit != 0; };
    for (int l = 0; l < L; ++l) {
        sp.eff[l] = layers[l]; sp.split[l] = false;
        sp.other[l] = other && other[l].kind != DPCLIP_KIND_DENSE;
        const size_t off0 = off;
        const int jobs0 = sp.n_jobs;
        if (sp.other[l]) {
            if (other[l].kind != DPCLIP_KIND_CONV) continue;
            const dpclip_layer& y = other[l].layer;
            const dpclip_conv& g = other[l].conv;
            SimtParams p;
            int T = 0;
            if (conv_setup(p, y.A, y.Zbar, other[l].z_channel_major, B, &g, y.d_out, dtype, y.has_bias, &T)) continue;
            if (T <= 1 || !y.gW || y.ldg != p.d_in || (y.has_bias && !y.gb)) continue;
            if (conv_tc_ok(p, y.A, y.Zbar, other[l].z_channel_major, B, T, dtype, base, kHeaderBytes)) continue;
            // bf16: the gathers of the fp32-ALU convolution kernel cost more than the copy from small sizes on (a CNN with
            // layers of 4 to 90 M multiply-adds: 80 us, 45 us staged)
            if ((double)B * T * p.d_in * p.d_out < (dtype == DPCLIP_BF16 ? 4.0 : 32.0) * 1024 * 1024) continue;
            // narrow fp32 layers go to the kernels that stream dense rows
            const bool narrow = dtype == DPCLIP_F32 && narrow_layer(T, p.d_in, p.d_out, 1, p.d_in, p.d_out);
            const long ldp = narrow ? p.d_in : (long)round_up(p.d_in, unit), ldz = narrow ? p.d_out : (long)round_up(p.d_out, unit);
            const int kk = g.kh * g.kw;
            if ((double)B * T * ldp / unit > 4.0e9 || g.kh > 16 || g.kw > 16) continue;
            // A CTA: about 144 columns in whole channels whose columns are a multiple of 16 bytes, and 32 to 256 positions, about 18432
            // elements in all: rows of positions of one example, or whole examples (9216 and 36864 elements, 288 and 576 columns:
            // up to 15 % slower on the layers of two CNNs).  Odd rows of a narrow layer take one block of all channels.
            stage::Job im;
            memset(&im, 0, sizeof(im));
            const int Ho = T / p.Wo;
            im.T = T; im.C = g.C; im.H = g.H; im.W = g.W; im.kh = g.kh; im.kw = g.kw; im.stride = g.stride; im.pad = g.pad; im.Wo = p.Wo;
            im.es = (int)es; im.dst_ld = (int)ldp; im.cols = p.d_in; im.rows = B * T;
            bool short_of_room = false;
            auto cut = [&](int ct, int positions) {
                im.ct = ct;
                im.n_ex = positions / T > 1 ? positions / T : 1;
                if (im.n_ex > B) im.n_ex = B;
                im.r_out = positions / p.Wo < 1 ? 1 : positions / p.Wo > Ho ? Ho : positions / p.Wo;
                im.tiles_a = ceil_div(Ho, (long)im.r_out); im.tiles_b = ceil_div(g.C, (long)ct);
                im.part = 0; im.w_out = p.Wo; im.tiles_x = 1; im.lead = 0; im.pitch = g.W + 2 * g.pad;
                // loads start at a channel's first valid row: a multiple of W elements, or the channel's start when a CTA takes it whole
                for (im.vec = unit; im.vec > 1; im.vec /= 2)
                    if (aligned_to(y.A, im.vec * es) && (g.H * g.W) % im.vec == 0 && (im.tiles_a == 1 || g.W % im.vec == 0)) break;
                if (p.Wo > kLongRow || (short_of_room && positions < p.Wo)) {
                    im.part = 1; im.r_out = 1; im.tiles_a = Ho; im.n_ex = 1;
                    im.w_out = ceil_div(p.Wo, ceil_div(p.Wo, (long)positions));
                    if (im.w_out > 8) im.w_out = (int)round_up(im.w_out, 8);
                    im.tiles_x = ceil_div(p.Wo, (long)im.w_out);
                    for (im.vec = unit; im.vec > 1; im.vec /= 2)
                        if (aligned_to(y.A, im.vec * es) && g.W % im.vec == 0 && (im.w_out * g.stride) % im.vec == 0) break;
                    im.lead = (im.vec - g.pad % im.vec) % im.vec;
                    im.pitch = (int)round_up(im.lead + (im.w_out - 1) * g.stride + g.kw, im.vec);
                }
                const double plane = ((im.r_out - 1.0) * g.stride + g.kh) * im.pitch;
                im.plane = plane < 1 << 20 ? (int)plane : 1 << 20;            // far beyond any limit either way
            };
            // whether the window, its channels apart on the banks, takes more than so many bytes
            auto above = [&](size_t limit) {
                if (stage::im_smem(im) > limit) return true;
                stage::Job widest = im;
                widest.plane += stage::IM_MAX_PAD;
                if (stage::im_smem(widest) <= limit) return false;
                widest.plane = im.plane + stage::im_bank_pad(im);
                return stage::im_smem(widest) > limit;
            };
            int ct = ldp % unit ? g.C : 144 / kk / unit * unit;
            if (ct < unit && ldp % unit == 0) ct = unit;
            if (ct > g.C) ct = g.C;
            int positions = 18432 / (ct * kk);
            positions = positions < 32 ? 32 : positions > 256 ? 256 : positions;
            cut(ct, positions);
            while (positions > 32 && (above(48 * 1024) || (long)ceil_div(B, (long)im.n_ex) * im.tiles_a * im.tiles_x * im.tiles_b < kNumSMs))
                cut(ct, positions /= 2);
            while (above(stage::SMEM_MAX)) {
                if (ct > unit && ldp % unit == 0) ct = (int)round_up((size_t)ct / 2, unit);
                else if (positions > 1) { short_of_room = true; positions /= 2; }
                else break;
                cut(ct, positions);
            }
            if (above(stage::SMEM_MAX) || (double)im.n_ex * g.C * g.H * g.W > 2.0e9) continue;
            im.plane += stage::im_bank_pad(im);
            const size_t im_bytes = stage::im_smem(im);
            {
                stage::Job& j = add_job(l, false, stage::IM2COL, y.A, 0, (int)ldp, B * T, p.d_in, es);
                im.kind = j.kind; im.src = j.src; im.src_ld = 0;
                j = im;
                if ((int)im_bytes > sp.smem) sp.smem = (int)im_bytes;
            }
            dpclip_layer& e = sp.eff[l];
            e = y;
            e.T = T; e.d_in = p.d_in; e.lda = ldp; e.method = DPCLIP_AUTO; e.ldz = p.d_out;
            if (other[l].z_channel_major) {
                stage::Job& j = add_job(l, true, stage::TRANSPOSE, y.Zbar, 0, (int)ldz, B * T, p.d_out, es);
                j.ct = p.d_out <= 32 ? 32 : 64;
                j.T = T; j.tiles_a = ceil_div(T, stage::TILE / j.ct); j.tiles_b = ceil_div(p.d_out, j.ct);
                const int bytes = j.ct * (stage::TILE / j.ct + 2) * (int)es;
                if (bytes > sp.smem) sp.smem = bytes;
                e.ldz = ldz;
            } else if (!narrow && misaligned(y.Zbar, p.d_out)) {
                add_job(l, true, stage::ROWS, y.Zbar, p.d_out, (int)ldz, B * T, p.d_out, es);
                e.ldz = ldz;
            }
        } else {
            const dpclip_layer& y = layers[l];
            if (y.T <= 1 || y.method != DPCLIP_AUTO || !y.gW || y.ldg != y.d_in || (y.has_bias && !y.gb)) continue;
            if (check_layer_args(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype)) continue;
            const bool sa = misaligned(y.A, y.lda), sz = misaligned(y.Zbar, y.ldz);
            if (!(sa || sz) || narrow_layer(y.T, y.d_in, y.d_out, y.has_bias, y.lda, y.ldz)) continue;
            if (!stage_worth_it((double)B * y.T, (double)y.d_in * y.d_out, dtype)) continue;
            if ((double)B * y.T * round_up(y.d_in > y.d_out ? y.d_in : y.d_out, unit) / unit > 4.0e9) continue;
            const long lda = (long)round_up(y.d_in, unit), ldz = (long)round_up(y.d_out, unit);
            if (sa) { add_job(l, false, stage::ROWS, y.A, y.lda, (int)lda, B * y.T, y.d_in, es); sp.eff[l].lda = lda; }
            if (sz) { add_job(l, true, stage::ROWS, y.Zbar, y.ldz, (int)ldz, B * y.T, y.d_out, es); sp.eff[l].ldz = ldz; }
        }
        if (off > kStageCapBytes) {                                  // does not fit: this layer stays as it is
            off = off0; sp.n_jobs = jobs0;
            sp.eff[l] = layers[l];
            continue;
        }
        sp.other[l] = false;
        sp.split[l] = dtype == DPCLIP_BF16;
        any = true;
    }
    // T = 1 layers taken together (see prepare_t1_group): one operand that TMA cannot address keeps all of them off the
    // tensor cores.  fp32: such operands are copied.  bf16: the operands of all of them become fp32 (the fp32-ALU kernel
    // that these models ran on before applies the factors in fp32; rounding them to bf16 would be a loss).
    if (t1_too && B <= FUSED_MAX_B && !path_switch(SW_NO_FUSED_T1) && !path_switch(SW_NO_T1_TF32)) {
        // Worth it from about 2e8 multiply-adds at B >= 64 in bf16, at B >= 256 in fp32 (whole steps, staged / not: B = 256,
        // 1001 -> 1001: 35 / 39 us, 2001: 64 / 115; B = 64, bf16, 2001: 51 / 58, 1001: 30 / 33; B = 64, fp32, 1001: 30 / 24;
        // B = 95, fp32, 475 M in five layers: 52 / 48; B = 16, 4001: 163 / 125).
        int n = 0, wide = 0;
        bool bad = false, ok = B >= (dtype == DPCLIP_BF16 ? 64 : 256);
        double macs = 0.0;
        for (int l = 0; l < L; ++l) {
            const dpclip_layer& y = layers[l];
            if (sp.other[l] || y.T != 1 || (other && other[l].kind != DPCLIP_KIND_DENSE)) continue;
            ++n;
            if (check_layer_args(y.A, y.lda, y.Zbar, y.ldz, B, 1, y.d_in, y.d_out, dtype)) { ok = false; break; }
            ok = ok && (y.method == DPCLIP_AUTO || y.method == DPCLIP_T1) && y.ldg == y.d_in && y.gW && aligned_to(y.gW, 16) &&
                 !(y.has_bias && !y.gb);
            const bool thin = y.d_out <= tc::f1::THIN_MAX_OUT;
            wide += !thin;
            macs += (double)B * y.d_in * y.d_out;
            bad = bad || misaligned(y.A, y.lda) || (!thin && misaligned(y.Zbar, y.ldz));
        }
        if (ok && bad && macs >= 2e8 && n > 0 && n <= FUSED_MAX_LAYERS && wide > 0) {
            const bool cvt = dtype == DPCLIP_BF16;
            const size_t off0 = off;
            const int jobs0 = sp.n_jobs;
            for (int l = 0; l < L; ++l) {
                const dpclip_layer& y = layers[l];
                if (sp.other[l] || y.T != 1 || (other && other[l].kind != DPCLIP_KIND_DENSE)) continue;
                const bool thin = y.d_out <= tc::f1::THIN_MAX_OUT;
                const long lda = (long)round_up(y.d_in, 4), ldz = (long)round_up(y.d_out, 4);
                if (cvt || misaligned(y.A, y.lda)) {
                    add_job(l, false, cvt ? stage::ROWS_TO_F32 : stage::ROWS, y.A, y.lda, (int)lda, B, y.d_in, 4);
                    sp.eff[l].lda = lda;
                }
                if (cvt || (!thin && misaligned(y.Zbar, y.ldz))) {
                    add_job(l, true, cvt ? stage::ROWS_TO_F32 : stage::ROWS, y.Zbar, y.ldz, (int)ldz, B, y.d_out, 4);
                    sp.eff[l].ldz = ldz;
                }
            }
            if (off > kStageCapBytes) {
                off = off0; sp.n_jobs = jobs0;
                for (int l = 0; l < L; ++l) if (!sp.other[l] && layers[l].T == 1) sp.eff[l] = layers[l];
            } else {
                any = true;
                sp.t1_dtype = DPCLIP_F32;
            }
        }
    }
    if (!any) return false;
    bool all_t1 = other == nullptr;
    for (int l = 0; l < L; ++l) all_t1 = all_t1 && sp.eff[l].T == 1;
    sp.scratch = round_up(step_scratch_bytes(sp.eff, L, B, dtype), 256);
    if (all_t1 && sp.t1_dtype != dtype) {                            // the planes of a model that has become fp32
        const size_t w = round_up(step_scratch_bytes(sp.eff, L, B, sp.t1_dtype), 256);
        if (w > sp.scratch) sp.scratch = w;
    }
    if (other) {
        for (int l = 0; l < L; ++l) {
            if (!sp.other[l] || other[l].kind != DPCLIP_KIND_CONV) continue;
            const size_t w = round_up(dpclip_conv_workspace_bytes(B, &other[l].conv, other[l].layer.d_out, dtype, other[l].z_channel_major), 256);
            if (w > sp.scratch) sp.scratch = w;
        }
    }
    sp.bytes = sp.scratch + off;
    for (int i = 0; i < sp.n_jobs; ++i) {
        char* dst = base + sp.scratch + takes[i].off;
        sp.job[i].dst = dst;
        (takes[i].z ? sp.eff[takes[i].layer].Zbar : sp.eff[takes[i].layer].A) = dst;
    }
    sp.active = true;
    return true;
}

static size_t staged_workspace_bytes(const dpclip_layer* layers, const dpclip_model_layer* other, int L, int B, dpclip_dtype dtype,
                                     bool with_copies) {
    if (!layers || L <= 0 || B <= 0) return 0;
    StagePlan sp;
    if (!stage_plan(sp, layers, other, L, B, dtype, reinterpret_cast<char*>(256), true)) return 0;
    return with_copies ? sp.bytes : sp.scratch;
}

// sq [n_sq]: cleared by the way
static int launch_stage(StagePlan& sp, float* sq, size_t n_sq, cudaStream_t st) {
    for (int i0 = 0; i0 < sp.n_jobs; i0 += stage::MAX_JOBS) {
        stage::Launch q;
        memset(&q, 0, sizeof(q));
        q.n = sp.n_jobs - i0 < stage::MAX_JOBS ? sp.n_jobs - i0 : stage::MAX_JOBS;
        if (i0 == 0) { q.clear = sq; q.n_clear = n_sq; }
        bool parts = false;
        for (int i = 0; i < q.n; ++i) {
            stage::Job& j = q.job[i] = sp.job[i0 + i];
            parts = parts || j.part;
            j.blk_begin = q.blocks;
            if (j.kind == stage::IM2COL) q.blocks += ceil_div((long)j.rows / j.T, (long)j.n_ex) * j.tiles_a * j.tiles_x * j.tiles_b;
            else if (j.kind == stage::TRANSPOSE) q.blocks += j.rows / j.T * j.tiles_a * j.tiles_b;
            else q.blocks += ceil_div((long)j.rows * (j.dst_ld / ((j.es == 4 || j.kind == stage::ROWS_TO_F32) ? 4 : 8)),
                                      (long)stage::ROWS_UNROLL * stage::THREADS);
        }
        // the limit is the kernel's, not the launch's: a smaller one would fail the launch another thread is about to make
        const auto kernel = parts ? stage_operands_kernel<true> : stage_operands_kernel<false>;
        if (sp.smem > 48 * 1024 && !enable_smem(kernel, stage::SMEM_MAX)) return DPCLIP_ERR_CUDA;
        kernel<<<q.blocks, stage::THREADS, sp.smem, st>>>(q);
        if (launch_status()) return DPCLIP_ERR_CUDA;
    }
    return DPCLIP_OK;
}

// The layers of a step that share the launches of launch_group: T > 1, addressable by TMA, not taken by another shared
// launch (skip), and -- for the norms -- by the materialised product.  taken[l] is set for them.
static bool group_candidate(const dpclip_layer& y, int B, dpclip_dtype dtype) {
    if (y.T <= 1 || check_layer_args(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype)) return false;
    return dtype == DPCLIP_F32 && tf32_eligible(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype) &&
           !narrow_layer(y.T, y.d_in, y.d_out, y.has_bias, y.lda, y.ldz);
}
// The layers that stay of the n taken: on several streams those that pay, of one or two fp32 layers the wide ones
static int keep_group(GroupLayer* g, int n, const dpclip_layer* layers, int L, int B, bool norm, int streams, int* taken) {
    auto keep = [&](auto&& stays) {
        int k = 0, i = 0;
        for (int l = 0; l < L; ++l) {
            if (!taken[l]) continue;
            if (stays(layers[l])) g[k++] = g[i]; else taken[l] = 0;
            ++i;
        }
        return k;
    };
    const int all = n;
    if (streams > 1) n = keep([&](const dpclip_layer& y) { return group_joins(y, B, all, norm); });
    if (n < kGroupFrom) n = keep([](const dpclip_layer& y) { return group_wide(y.d_in, y.d_out); });
    return n;
}
struct NormGroup {
    GroupLayer g[64];
    int n = 0;
};
static int norm_group_layers(NormGroup& q, const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float* sq_layers, const int* skip,
                             int* taken, const void* workspace, size_t workspace_bytes, int streams) {
    q.n = 0;
    for (int l = 0; l < L; ++l) {
        taken[l] = 0;
        const dpclip_layer& y = layers[l];
        if ((skip && skip[l]) || !group_candidate(y, B, dtype)) continue;
        int method = y.method;
        if (method == DPCLIP_AUTO) method = dpclip_pick_method(B, y.T, y.d_in, y.d_out, y.lda, y.ldz, dtype);
        if (method != DPCLIP_MATERIALIZE) continue;
        q.g[q.n++] = {y.A, y.lda, y.Zbar, y.ldz, y.T, y.d_in, y.d_out, y.has_bias != 0, sq_layers + (size_t)l * B};
        taken[l] = 1;
    }
    q.n = keep_group(q.g, q.n, layers, L, B, true, streams, taken);
    if (q.n == 0) return DPCLIP_OK;
    if (!workspace || workspace_bytes < (size_t)kHeaderBytes) return DPCLIP_ERR_WORKSPACE;
    if (!group_norm_room(q.g, q.n, workspace_bytes)) {                                   // layer by layer
        q.n = 0;
        for (int l = 0; l < L; ++l) taken[l] = 0;
    }
    return DPCLIP_OK;
}
static int launch_norm_group(const NormGroup& q, int L, int B, void* workspace, size_t workspace_bytes, void* stream,
                             const tc::gram::FactorsTail* tail, bool* tail_done) {
    if (q.n == 0) return DPCLIP_OK;
    const bool with_tail = tail && q.n == L;
    if (tail_done) *tail_done = with_tail;
    return launch_group(q.g, q.n, B, true, nullptr, nullptr, workspace, workspace_bytes, (cudaStream_t)stream, with_tail ? tail : nullptr);
}
// clip_ld as in shared_clipped_grad_launches
static int group_grads(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, const float* clip, long clip_ld,
                       float C, float sigma, unsigned long long seed, unsigned long long stream_id0, const int* skip, int* taken,
                       void* workspace, size_t workspace_bytes, void* stream, int streams) {
    GroupLayer g[64];
    int n = 0;
    for (int l = 0; l < L; ++l) {
        taken[l] = 0;
        const dpclip_layer& y = layers[l];
        if ((skip && skip[l]) || !group_candidate(y, B, dtype) || !y.gW || y.ldg != y.d_in || (y.has_bias && !y.gb)) continue;
        g[n++] = {y.A, y.lda, y.Zbar, y.ldz, y.T, y.d_in, y.d_out, false, nullptr, clip ? clip + (size_t)l * clip_ld : nullptr,
                  y.gW, y.ldg, y.has_bias ? y.gb : nullptr, stream_id0 + 2ull * l, stream_id0 + 2ull * l + 1};
        taken[l] = 1;
    }
    n = keep_group(g, n, layers, L, B, false, streams, taken);
    if (n == 0) return DPCLIP_OK;
    const NoiseSpec ns = {sigma * C, seed, 0, 0};
    bool noise_done = false;
    const int rc = launch_group(g, n, B, false, &ns, &noise_done, workspace, workspace_bytes, (cudaStream_t)stream);
    if (rc > 0) { for (int l = 0; l < L; ++l) taken[l] = 0; return DPCLIP_OK; }         // no room: layer by layer
    return rc;
}

// The streams a step may spread its layers over.  Lane 0 is the caller's stream: the step starts and ends
// there.  fork() makes every other lane wait for what lane 0 has enqueued so far, join() makes lane 0 wait for
// what the other lanes have enqueued; both are event record/wait pairs, which a stream capture records as
// graph dependencies.  Every lane has a workspace of its own (launches on different lanes may overlap).
struct Lanes {
    static constexpr int kMax = 8;
    int n = 1;
    cudaStream_t st[kMax] = {};
    void* ws[kMax] = {};
    size_t ws_bytes[kMax] = {};
    cudaEvent_t ev[2 * kMax + 2] = {};
    int n_ev = 0;
    ~Lanes() { for (int i = 0; i < n_ev; ++i) cudaEventDestroy(ev[i]); }     // pending work keeps what it needs
    // events are reused between the fork and the join of a stage: a record replaces the earlier one for later waits only
    int event(cudaEvent_t* out) {
        if (n_ev == 2 * kMax + 2) return DPCLIP_ERR_CUDA;
        if (cudaEventCreateWithFlags(&ev[n_ev], cudaEventDisableTiming) != cudaSuccess) return DPCLIP_ERR_CUDA;
        *out = ev[n_ev++];
        return DPCLIP_OK;
    }
    int fork() {
        if (n == 1) return DPCLIP_OK;
        cudaEvent_t e;
        if (event(&e)) return DPCLIP_ERR_CUDA;
        if (cudaEventRecord(e, st[0]) != cudaSuccess) return DPCLIP_ERR_CUDA;
        for (int i = 1; i < n; ++i)
            if (cudaStreamWaitEvent(st[i], e, 0) != cudaSuccess) return DPCLIP_ERR_CUDA;
        return DPCLIP_OK;
    }
    int join() {
        for (int i = 1; i < n; ++i) {
            cudaEvent_t e;
            if (event(&e)) return DPCLIP_ERR_CUDA;
            if (cudaEventRecord(e, st[i]) != cudaSuccess || cudaStreamWaitEvent(st[0], e, 0) != cudaSuccess)
                return DPCLIP_ERR_CUDA;
        }
        return DPCLIP_OK;
    }
};

// The path layer by layer (with the launches that several layers share), Algorithm 1's order: every layer's
// norms, then the factors, then every layer's clipped sum with its noise.  Layers are independent within the
// norm stage and within the clipped-sum stage, so with several lanes the launches of a stage are dealt to the
// lanes (a layer's kernel then starts on SMs the previous layer's kernel has already left): the shared Gram
// launch and the shared same-shape launch on lane 0, the T = 1 group on the last lane, the rest round-robin.
// `other`, when given, is the model's own descriptor array: entries of a kind other than dense have a
// placeholder with T = 0 in `layers`, which every grouping rule below passes over, and go through the two
// functions above.
static int step_general(const dpclip_layer* layers_in, const dpclip_model_layer* other, int L, int B, dpclip_dtype dtype,
                        float C, float sigma, unsigned long long seed, unsigned long long stream_id0,
                        float* sq_layers, float* clip, float* norms, Lanes& lanes, StagePlan* sp, float* const* ew_rows = nullptr) {
    int rc;
    const dpclip_layer* layers = sp ? sp->eff : layers_in;              // the layers with their staged operands
    dpclip_dtype t1_dtype = sp ? sp->t1_dtype : dtype;
    const bool* split = sp ? sp->split : nullptr;
    auto other_kind = [&](int l) { return sp ? sp->other[l] : (other && other[l].kind != DPCLIP_KIND_DENSE); };
    bool any_other = false;
    for (int l = 0; l < L; ++l) any_other = any_other || other_kind(l);
    const int last = lanes.n - 1;
    void* const ws0 = lanes.ws[0];
    T1Group t1;
    rc = prepare_t1_group(t1, layers, L, B, t1_dtype, C, sigma, seed, stream_id0, sq_layers, clip);
    if (rc) return rc;
    if (t1.active && (!lanes.ws[last] || lanes.ws_bytes[last] < (size_t)kHeaderBytes)) t1.active = false;
    if (!t1.active && sp && t1_dtype != dtype) {                        // not taken together after all: the inputs as given
        for (int l = 0; l < L; ++l) if (layers_in[l].T == 1) sp->eff[l] = layers_in[l];
        t1_dtype = dtype;
    }
    // The rows of sq that launches add up with atomics: cleared by the staging launch, else on several streams all at once in
    // front of the fork.
    bool cleared = sp != nullptr;
    if (!cleared && lanes.n > 1) {
        const size_t n = (size_t)L * B;
        clear_kernel<<<(unsigned)(n < 256 * 64 ? (n + 255) / 256 : 64), 256, 0, lanes.st[0]>>>(sq_layers, n);
        if (cudaGetLastError() != cudaSuccess) return DPCLIP_ERR_CUDA;     // not in the count of launches, like the memsets it stands for
        cleared = true;
    }
    if ((rc = lanes.fork())) return rc;
    if (t1.active) {
        if (t1_dtype == DPCLIP_F32) t1_all_norms_kernel<float><<<t1.p.L * B, 128, 0, lanes.st[last]>>>(t1.p);
        else t1_all_norms_kernel<__nv_bfloat16><<<t1.p.L * B, 128, 0, lanes.st[last]>>>(t1.p);
        if (launch_status()) return DPCLIP_ERR_CUDA;
    }
    int in_gram_group[64];
    const bool track = L <= 64;
    bool any_gram = false, any_mat = false;
    bool factors_done = false;
    SqClearedScope cleared_scope(cleared);
    // when one launch takes every layer of the model, its last CTA also computes the factors
    const tc::gram::FactorsTail tail = {sq_layers, L, (long)B, B, C, clip, norms, nullptr, 0, {}};
    NormGroup norm_group;
    int mat_lane = 0;
    auto launch_mat_norms = [&]() {
        return launch_norm_group(norm_group, L, B, lanes.ws[mat_lane], lanes.ws_bytes[mat_lane], lanes.st[mat_lane],
                                 (!t1.active && !any_other && !any_gram && !path_switch(SW_NO_FACTORS_TAIL)) ? &tail : nullptr,
                                 any_gram ? nullptr : &factors_done);
    };
    if (track) {
        const OverlapPrevScope behind_copies(sp != nullptr && lanes.n == 1);
        rc = gram_layers_sqnorms(layers, L, B, dtype, sq_layers, in_gram_group, ws0, lanes.ws_bytes[0], lanes.st[0],
                                 (!t1.active && !any_other && !path_switch(SW_NO_FACTORS_TAIL)) ? &tail : nullptr, &factors_done);
        if (rc) return rc;
        for (int l = 0; l < L; ++l) any_gram = any_gram || in_gram_group[l];
        // the layers whose norms go by the materialised product, also in one launch
        int skip[64], taken[64];
        for (int l = 0; l < L; ++l) skip[l] = in_gram_group[l] || other_kind(l);
        mat_lane = any_gram && lanes.n > 1 ? 1 : 0;
        rc = norm_group_layers(norm_group, layers, L, B, dtype, sq_layers, skip, taken, lanes.ws[mat_lane], lanes.ws_bytes[mat_lane], lanes.n);
        if (rc) return rc;
        for (int l = 0; l < L; ++l) {
            any_mat = any_mat || taken[l];
            if (taken[l]) in_gram_group[l] = 1;                          // nothing left to do for it in this stage
        }
        if (lanes.n == 1 && (rc = launch_mat_norms())) return rc;
    }
    // SM shares for the per-layer launches of a stage (see t_sm_budget): only when several of them run side by
    // side on different lanes, no launch shared by several layers is in the stage, and the stage is small
    const size_t es = elt_size(dtype);
    auto layer_bytes = [&](int l) -> double {
        if (other_kind(l) && other[l].kind == DPCLIP_KIND_CONV) {
            const dpclip_conv& g = other[l].conv;
            const double Ho = (g.H + 2 * g.pad - g.kh) / g.stride + 1, Wo = (g.W + 2 * g.pad - g.kw) / g.stride + 1;
            return (double)B * ((double)g.C * g.H * g.W + Ho * Wo * other[l].layer.d_out) * es;
        }
        const dpclip_layer& y = other_kind(l) ? other[l].layer : layers[l];
        return (double)B * y.T * ((double)y.d_in + y.d_out) * es;
    };
    auto stage_budgets = [&](const int* skip, bool shared_launch, int* budget) {
        int n_ent = 0;
        double total = 0.0;
        for (int l = 0; l < L; ++l) {
            budget[l] = 0;
            const bool is_other = other_kind(l);
            if (!is_other && ((t1.active && layers[l].T == 1) || (skip && skip[l]))) continue;
            ++n_ent; total += layer_bytes(l);
        }
        // bf16 only: the fp32 forms (three tf32 MMAs per product, four operand planes to prepare, gathers) are
        // bound by their own work, and a share of the SMs stretches them in proportion (measured: the feature-map
        // CNN in fp32 242 -> 312 us with shares, in bf16 98 -> 86 us; the patch-matrix CNN in bf16 94 -> 79 us)
        if (dtype != DPCLIP_BF16 || lanes.n < 2 || n_ent < 2 || shared_launch || total > 400e6 ||
            path_switch(SW_NO_SM_BUDGET)) return;
        const double widen = n_ent > lanes.n ? (double)n_ent / lanes.n : 1.0;      // more launches than lanes: some queue
        for (int l = 0; l < L; ++l) {
            const bool is_other = other_kind(l);
            if (!is_other && ((t1.active && layers[l].T == 1) || (skip && skip[l]))) continue;
            int b = (int)(kNumSMs * layer_bytes(l) / total * widen + 0.5);
            budget[l] = b < 16 ? 16 : (b > kNumSMs ? kNumSMs : b);
        }
    };
    int budget[64] = {0};
    if (track) stage_budgets(in_gram_group, any_gram || any_mat, budget);
    auto alone = [&](int l) { return other_kind(l) || !((t1.active && layers[l].T == 1) || (track && in_gram_group[l])); };
    // The shared fp32 kernel fills every SM, so what stands beside it starts first, from this stream: behind it a layer of 18 CTAs on the
    // fp32 ALUs (18 examples of 28 x 28 maps, 3 -> 64 channels, beside 64 -> 256 -> 256 -> 256) began when it was over, 342 us a step instead of 268.
    bool beside = false;
    for (int l = 0; l < L; ++l) beside = beside || alone(l);
    if (any_mat && !any_gram && beside && lanes.n > 1 && lanes.ws[1] && group_norm_room(norm_group.g, norm_group.n, lanes.ws_bytes[1])) mat_lane = 1;
    const bool moved = mat_lane == 1 && !any_gram;
    int k = moved ? 0 : (any_gram ? 1 : 0) + (any_mat ? 1 : 0);        // the first lanes already carry the shared launches
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        if (!alone(l)) continue;
        const bool is_other = other_kind(l);
        const SmBudgetScope share(track ? budget[l] : 0);
        const int i = k++ % lanes.n, b = !moved || i == 0 ? i : i == lanes.n - 1 ? 1 : i + 1;      // moved: 0, 2, 3, ..., 1
        if (is_other)
            rc = other_kind_sqnorms(other[l], B, dtype, sq_layers + (size_t)l * B, ew_rows ? ew_rows[l] : nullptr, lanes.ws[b],
                                    lanes.ws_bytes[b], lanes.st[b]);
        else
            rc = dpclip_layer_sqnorms(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype, y.has_bias,
                                      (dpclip_method)y.method, sq_layers + (size_t)l * B, lanes.ws[b],
                                      lanes.ws_bytes[b], lanes.st[b]);
        if (rc) return rc;
    }
    if (lanes.n > 1 && (rc = launch_mat_norms())) return rc;
    if ((rc = lanes.join())) return rc;
    if (!factors_done) {
        // on one stream right behind the last of the norms
        if (lanes.n == 1)
            rc = launch_behind(factors_kernel, dim3(1), 256, 0, lanes.st[0], (const float*)sq_layers, L, (long)B, B, C, clip, norms, (int*)nullptr);
        else
            rc = dpclip_factors(sq_layers, L, B, B, C, clip, norms, nullptr, lanes.st[0]);
        if (rc) return rc;
    }
    if ((rc = lanes.fork())) return rc;
    auto t1_grads = [&]() -> int {
        const int r = t1.active ? launch_fused_t1_tf32(t1.p, false, t1_dtype, lanes.ws[last], lanes.ws_bytes[last], lanes.st[last]) : 0;
        return r > 0 ? DPCLIP_ERR_UNSUPPORTED : r;           // prepare_t1_group checked the same conditions
    };
    // fp32 on several streams: behind the other sums of its stream.  Steps of two CNNs, first / last: 132.8 / 129.9 and 162.2 / 160.2 us, with inputs
    // from HBM 141.1 / 139.7 and 170.3 / 168.0.  (bf16 was measured first: a CNN's launch of 12 us beside three longer ones.)
    const bool t1_last = dtype == DPCLIP_F32 && lanes.n > 1;
    if (!t1_last && (rc = t1_grads())) return rc;
    int in_grad_group[64];
    bool any_group = false, any_rest = false;
    if (track) {
        // the factors came from the tail of the Gram launch or from factors_kernel, the last kernel of this stream: the first
        // clipped-sum launch may start loading while that runs
        const OverlapPrevScope overlap(factors_done || lanes.n == 1);
        // Layers of several T would share several launches, one after the other on lane 0, where side by side on the lanes they
        // are faster (four convolutions of 49 and 16 positions, 78 examples, four lanes: 68 us, 47 apart; layers of 100 and 50
        // positions: 70, 45).  On one lane sharing would win (77 us, 117 apart), but the shared kernel rounds c a where the
        // layers' own round c zb, and a step's results do not depend on the number of lanes.
        bool join = true;
        int T_dense = 0;
        for (int l = 0; l < L; ++l) {
            if (other_kind(l) || layers[l].T <= 1) continue;
            join = join && (T_dense == 0 || layers[l].T == T_dense);
            T_dense = layers[l].T;
        }
        rc = shared_clipped_grad_launches(layers, split, join, L, B, dtype, clip, 0, C, sigma, seed, stream_id0, in_grad_group, ws0,
                                          lanes.ws_bytes[0], lanes.st[0]);
        if (rc) return rc;
        for (int l = 0; l < L; ++l) any_group = any_group || in_grad_group[l];
        int skip[64], taken[64];
        for (int l = 0; l < L; ++l) skip[l] = in_grad_group[l] || other_kind(l) || (t1.active && layers[l].T == 1);
        const int b = any_group && lanes.n > 1 ? 1 : 0;
        rc = group_grads(layers, L, B, dtype, clip, 0, C, sigma, seed, stream_id0, skip, taken, lanes.ws[b], lanes.ws_bytes[b],
                         lanes.st[b], lanes.n);
        if (rc) return rc;
        for (int l = 0; l < L; ++l) if (taken[l]) { any_rest = true; in_grad_group[l] = 1; }
    }
    if (track) stage_budgets(in_grad_group, any_group || any_rest, budget);
    k = (any_group ? 1 : 0) + (any_rest ? 1 : 0);
    // On several streams the small layers of one position go first, on the last one: a few microseconds in front of that stream's
    // larger layer, where at their place in the order they ended the stage.
    auto first = [&](int l) { return lanes.n > 1 && !other_kind(l) && t1_thin_ok(layers[l].A, layers[l].lda, B, layers[l].T, layers[l].d_in, layers[l].d_out, dtype); };
    if (ew_rows) {
        rc = ew_rows_grads(other, ew_rows, L, B, clip, C, sigma, seed, stream_id0, lanes.st[k % lanes.n]);
        if (rc) return rc;
        ++k;
    }
    for (int pass = lanes.n > 1 ? 0 : 1; pass < 2; ++pass)
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        const bool is_other = other_kind(l);
        if (!is_other && ((t1.active && y.T == 1) || (track && in_grad_group[l]))) continue;
        if (ew_rows && ew_rows[l]) continue;
        if (first(l) != (pass == 0)) continue;
        const SmBudgetScope share(track ? budget[l] : 0);
        const int b = pass == 0 ? last : k++ % lanes.n;
        void* const stream = lanes.st[b];
        void* const workspace = lanes.ws[b];
        const size_t workspace_bytes = lanes.ws_bytes[b];
        if (is_other) {
            rc = other_kind_clipped_grad_noise(other[l], B, dtype, clip, C, sigma, seed, stream_id0 + 2ull * l,
                                               stream_id0 + 2ull * l + 1, workspace, workspace_bytes, stream);
            if (rc) return rc;
            continue;
        }
        float* gb = y.has_bias ? y.gb : nullptr;
        if (y.has_bias && !gb) return DPCLIP_ERR_INVALID_ARG;
        // noise indexes the dense d_out x d_in tensor, so the step wants unpadded output rows
        if (y.ldg != y.d_in) return DPCLIP_ERR_UNSUPPORTED;
        rc = check_layer_args(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype);
        if (rc) return rc;
        if (!y.gW) return DPCLIP_ERR_INVALID_ARG;
        NoiseSpec ns = {sigma * C, seed, stream_id0 + 2ull * l, stream_id0 + 2ull * l + 1};
        bool noise_done = false;
        rc = clipped_grad_impl(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype, clip, y.gW, y.ldg, gb,
                               workspace, workspace_bytes, &ns, &noise_done, (cudaStream_t)stream, split && split[l]);
        if (rc) return rc;
        if (!noise_done) {
            rc = dpclip_add_noise(y.gW, (size_t)y.d_out * y.d_in, sigma, C, seed, ns.sid_w, stream);
            if (rc) return rc;
            if (gb) {
                rc = dpclip_add_noise(gb, (size_t)y.d_out, sigma, C, seed, ns.sid_b, stream);
                if (rc) return rc;
            }
        }
    }
    if (t1_last && (rc = t1_grads())) return rc;
    return lanes.join();
}

// Lanes of a one-stream call, and of a several-streams call (argument checks included).
static void one_lane(Lanes& lanes, void* workspace, size_t workspace_bytes, void* stream) {
    lanes.n = 1; lanes.st[0] = (cudaStream_t)stream; lanes.ws[0] = workspace; lanes.ws_bytes[0] = workspace_bytes;
}
// sizes: bytes of every lane's workspace, or NULL: workspace_bytes each
static int many_lanes(Lanes& lanes, int n_streams, void* const* streams, void* const* workspaces, const size_t* sizes,
                      size_t workspace_bytes) {
    if (n_streams < 1 || n_streams > Lanes::kMax || !streams || !workspaces) return DPCLIP_ERR_INVALID_ARG;
    lanes.n = n_streams;
    for (int i = 0; i < n_streams; ++i) {
        lanes.st[i] = (cudaStream_t)streams[i]; lanes.ws[i] = workspaces[i];
        lanes.ws_bytes[i] = sizes ? sizes[i] : workspace_bytes;
        for (int j = 0; j < i; ++j)
            if (streams[i] == streams[j] || (workspaces[i] && workspaces[i] == workspaces[j])) return DPCLIP_ERR_INVALID_ARG;
    }
    return DPCLIP_OK;
}

static int step_args_ok(const void* layers, int L, int B, dpclip_dtype dtype, float C, float sigma, const float* sq_layers,
                        const float* clip) {
    if (!layers || L <= 0 || B <= 0 || !sq_layers || !clip) return DPCLIP_ERR_INVALID_ARG;
    if (!(C > 0.f) || !(sigma >= 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (dtype != DPCLIP_F32 && dtype != DPCLIP_BF16) return DPCLIP_ERR_INVALID_ARG;
    return DPCLIP_OK;
}

// Plans and launches the staging of a step when the workspace has room for the copies (sp.active says so); the
// lanes' scratch then ends where the copies begin.
static int stage_step(StagePlan& sp, const dpclip_layer* layers, const dpclip_model_layer* other, int L, int B,
                      dpclip_dtype dtype, float* sq_layers, Lanes& lanes, bool t1_too) {
    if (!lanes.ws[0] || !stage_plan(sp, layers, other, L, B, dtype, static_cast<char*>(lanes.ws[0]), t1_too)) return DPCLIP_OK;
    if (lanes.ws_bytes[0] < sp.bytes) { sp.active = false; return DPCLIP_OK; }
    lanes.ws_bytes[0] = sp.scratch;                            // the copies lie behind lane 0's scratch
    return launch_stage(sp, sq_layers, (size_t)L * B, lanes.st[0]);
}

static int step_dense(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                      unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                      float* norms, Lanes& lanes) {
    StagePlan sp;
    int rc = stage_step(sp, layers, nullptr, L, B, dtype, sq_layers, lanes, true);
    if (rc) return rc;
    rc = try_fused_t1_step(sp.active ? sp.eff : layers, L, B, sp.active ? sp.t1_dtype : dtype, C, sigma, seed, stream_id0,
                           sq_layers, clip, norms, lanes.ws[0], lanes.ws_bytes[0], lanes.st[0]);
    if (rc <= 0) return rc;                  // done (0) or argument error (< 0); 1 = take the general path
    return step_general(layers, nullptr, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes,
                        sp.active ? &sp : nullptr);
}

// Scratch of a step over these layers, copies and per-example gradients aside; dense: the layers with T = 0 for other kinds.
static size_t model_scratch_bytes(const dpclip_model_layer* layers, const dpclip_layer* dense, int L, int B, dpclip_dtype dtype) {
    size_t ws = step_scratch_bytes(dense, L, B, dtype);
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l].layer;
        size_t w = kHeaderBytes;
        if (layers[l].kind == DPCLIP_KIND_DENSE)
            w = dpclip_workspace_bytes(B, y.T, y.d_in, y.d_out, dtype, (dpclip_method)y.method);
        else if (layers[l].kind == DPCLIP_KIND_CONV)
            w = dpclip_conv_workspace_bytes(B, &layers[l].conv, y.d_out, dtype, layers[l].z_channel_major);
        if (w > ws) ws = w;
    }
    return ws;
}

static int step_model(const dpclip_model_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                      unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                      float* norms, Lanes& lanes) {
    constexpr int kMaxLayers = 256;
    if (L > kMaxLayers) return DPCLIP_ERR_INVALID_ARG;
    dpclip_layer dense[kMaxLayers];
    bool all_dense = true;
    for (int l = 0; l < L; ++l) {
        if (layers[l].kind == DPCLIP_KIND_DENSE) { dense[l] = layers[l].layer; continue; }
        if (layers[l].kind != DPCLIP_KIND_ELEMENTWISE && layers[l].kind != DPCLIP_KIND_CONV) return DPCLIP_ERR_INVALID_ARG;
        memset(&dense[l], 0, sizeof(dense[l]));             // T = 0: no grouping rule takes it
        all_dense = false;
    }
    if (all_dense) return step_dense(dense, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes);
    StagePlan sp;
    const size_t given = lanes.ws_bytes[0];
    const int rc = stage_step(sp, dense, layers, L, B, dtype, sq_layers, lanes, true);
    if (rc) return rc;
    // the per-example gradients of the element-wise layers lie at the end of lane 0's workspace when it has room for them
    float* rows[kMaxLayers];
    const size_t ew = ew_rows_total(layers, L, B);
    bool use_rows = ew > 0 && lanes.ws[0] && given >= ew;
    if (use_rows) {
        size_t at = (given - ew) / 256 * 256;
        use_rows = at >= (sp.active ? sp.bytes : model_scratch_bytes(layers, dense, L, B, dtype));
        if (use_rows && lanes.ws_bytes[0] > at) lanes.ws_bytes[0] = at;
        for (int l = 0; use_rows && l < L; ++l) {
            const dpclip_layer& y = layers[l].layer;
            const size_t n = ew_rows_bytes(layers[l], B);
            rows[l] = nullptr;
            if (n == 0) continue;
            // the checks of dpclip_elementwise_clipped_grad
            if (!y.gW || (y.has_bias && !y.gb)) return DPCLIP_ERR_INVALID_ARG;
            if (!aligned_to(y.gW, 4) || (y.has_bias && !aligned_to(y.gb, 4))) return DPCLIP_ERR_MISALIGNED;
            rows[l] = reinterpret_cast<float*>(static_cast<char*>(lanes.ws[0]) + at);
            at += n;
        }
    }
    return step_general(dense, layers, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes,
                        sp.active ? &sp : nullptr, use_rows ? rows : nullptr);
}

int dpclip_step(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                float* norms, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = step_args_ok(layers, L, B, dtype, C, sigma, sq_layers, clip);
    if (rc) return rc;
    Lanes lanes;
    one_lane(lanes, workspace, workspace_bytes, stream);
    return step_dense(layers, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes);
}

int dpclip_step_streams(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                        unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                        float* norms, int n_streams, void* const* streams, void* const* workspaces,
                        size_t workspace_bytes) {
    int rc = step_args_ok(layers, L, B, dtype, C, sigma, sq_layers, clip);
    if (rc) return rc;
    Lanes lanes;
    if ((rc = many_lanes(lanes, n_streams, streams, workspaces, nullptr, workspace_bytes))) return rc;
    return step_dense(layers, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes);
}

int dpclip_step_lanes(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                        unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                        float* norms, int n_streams, void* const* streams, void* const* workspaces,
                        const size_t* workspace_bytes) {
    if (!workspace_bytes) return DPCLIP_ERR_INVALID_ARG;
    int rc = step_args_ok(layers, L, B, dtype, C, sigma, sq_layers, clip);
    if (rc) return rc;
    Lanes lanes;
    if ((rc = many_lanes(lanes, n_streams, streams, workspaces, workspace_bytes, 0))) return rc;
    return step_dense(layers, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes);
}

int dpclip_step_per_layer(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, const float* C_layer,
                          float sigma, unsigned long long seed, unsigned long long stream_id0, float* sq_layers,
                          float* clip_layers, float* norms_layers, void* workspace, size_t workspace_bytes,
                          void* stream) {
    if (!layers || L <= 0 || B <= 0 || !C_layer || !sq_layers || !clip_layers) return DPCLIP_ERR_INVALID_ARG;
    if (!(sigma >= 0.f)) return DPCLIP_ERR_INVALID_ARG;
    if (dtype != DPCLIP_F32 && dtype != DPCLIP_BF16) return DPCLIP_ERR_INVALID_ARG;
    double c2 = 0.0;
    for (int l = 0; l < L; ++l) {
        if (!(C_layer[l] > 0.f)) return DPCLIP_ERR_INVALID_ARG;
        c2 += (double)C_layer[l] * C_layer[l];
    }
    const float C_total = (float)sqrt(c2);               // sensitivity of the concatenated clipped gradient
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        if (!y.gW || (y.has_bias && !y.gb)) return DPCLIP_ERR_INVALID_ARG;
        if (y.ldg != y.d_in) return DPCLIP_ERR_UNSUPPORTED;            // noise indexes the dense tensor
    }
    int rc;
    // The stages of the global step with a factor vector per layer: every layer's norms (the layers that go by
    // the Gram identity in one launch), then ALL rows of factors in one launch (row l against C_layer[l]), then
    // the clipped sums -- the wide bf16 layers of one T in one CTA-pair launch, each with its own factor row --
    // with the noise N(0, sigma^2 * sum_l C_l^2).  (Layer after layer, norm -> factors -> clipped sum, so that a
    // layer's second pass finds its inputs in L2, took 566 us on the sequence workload: it gives up both shared
    // launches, and a wide layer's inputs do not fit L2 anyway.)
    constexpr int kMaxTracked = 64;
    int in_gram[kMaxTracked], in_pairs[kMaxTracked];
    const bool track = L <= kMaxTracked;
    StagePlan sp;
    {
        Lanes lanes;
        one_lane(lanes, workspace, workspace_bytes, stream);
        if ((rc = stage_step(sp, layers, nullptr, L, B, dtype, sq_layers, lanes, false))) return rc;
        workspace_bytes = lanes.ws_bytes[0];
    }
    const bool* split = sp.active ? sp.split : nullptr;
    if (sp.active) layers = sp.eff;
    bool factors_done = false;
    {
    const SqClearedScope cleared(sp.active);                            // by the staging launch
    if (track) {
        // when one launch takes every layer, its last CTA computes the factors too
        tc::gram::FactorsTail tail = {sq_layers, L, (long)B, B, 0.f, clip_layers, norms_layers, nullptr, 1, {}};
        const bool with_tail = L <= (int)(sizeof(tail.C_row) / sizeof(float)) && !path_switch(SW_NO_FACTORS_TAIL);
        for (int l = 0; with_tail && l < L; ++l) tail.C_row[l] = C_layer[l];
        const OverlapPrevScope behind_copies(sp.active);
        rc = gram_layers_sqnorms(layers, L, B, dtype, sq_layers, in_gram, workspace, workspace_bytes, stream, with_tail ? &tail : nullptr, &factors_done);
        if (rc) return rc;
        int taken[kMaxTracked];
        bool any_gram = false;
        for (int l = 0; l < L; ++l) any_gram = any_gram || in_gram[l];
        NormGroup norm_group;
        rc = norm_group_layers(norm_group, layers, L, B, dtype, sq_layers, in_gram, taken, workspace, workspace_bytes, 1);
        if (!rc) rc = launch_norm_group(norm_group, L, B, workspace, workspace_bytes, stream, with_tail && !any_gram ? &tail : nullptr,
                                        any_gram ? nullptr : &factors_done);
        if (rc) return rc;
        for (int l = 0; l < L; ++l) in_gram[l] = in_gram[l] || taken[l];
    }
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        if (track && in_gram[l]) continue;
        rc = dpclip_layer_sqnorms(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype, y.has_bias,
                                  (dpclip_method)y.method, sq_layers + (size_t)l * B, workspace, workspace_bytes, stream);
        if (rc) return rc;
    }
    }
    if (track) {
        if (!factors_done) {
            LayerThresholds th;
            for (int l = 0; l < L; ++l) th.C[l] = C_layer[l];
            if (launch_behind(factors_rows_kernel, dim3(L), 256, 0, (cudaStream_t)stream, (const float*)sq_layers, (long)B, B, th, clip_layers,
                              norms_layers)) return DPCLIP_ERR_CUDA;
        }
        const OverlapPrevScope overlap(true);
        rc = shared_clipped_grad_launches(layers, split, true, L, B, dtype, clip_layers, (long)B, C_total, sigma, seed, stream_id0,
                                          in_pairs, workspace, workspace_bytes, stream);
        if (rc) return rc;
        int taken[kMaxTracked];
        rc = group_grads(layers, L, B, dtype, clip_layers, (long)B, C_total, sigma, seed, stream_id0, in_pairs, taken, workspace,
                         workspace_bytes, stream, 1);
        if (rc) return rc;
        for (int l = 0; l < L; ++l) in_pairs[l] = in_pairs[l] || taken[l];
    } else {
        for (int l = 0; l < L; ++l) {
            rc = dpclip_factors(sq_layers + (size_t)l * B, 1, B, B, C_layer[l], clip_layers + (size_t)l * B,
                                norms_layers ? norms_layers + (size_t)l * B : nullptr, nullptr, stream);
            if (rc) return rc;
        }
    }
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        if (track && in_pairs[l]) continue;
        float* gb = y.has_bias ? y.gb : nullptr;
        NoiseSpec ns = {sigma * C_total, seed, stream_id0 + 2ull * l, stream_id0 + 2ull * l + 1};
        bool noise_done = false;
        rc = clipped_grad_impl(y.A, y.lda, y.Zbar, y.ldz, B, y.T, y.d_in, y.d_out, dtype, clip_layers + (size_t)l * B, y.gW,
                               y.ldg, gb, workspace, workspace_bytes, &ns, &noise_done, (cudaStream_t)stream, split && split[l]);
        if (rc) return rc;
        if (!noise_done) {
            rc = dpclip_add_noise(y.gW, (size_t)y.d_out * y.d_in, sigma, C_total, seed, ns.sid_w, stream);
            if (rc) return rc;
            if (gb) {
                rc = dpclip_add_noise(gb, (size_t)y.d_out, sigma, C_total, seed, ns.sid_b, stream);
                if (rc) return rc;
            }
        }
    }
    return DPCLIP_OK;
}

static size_t model_workspace_bytes(const dpclip_model_layer* layers, int L, int B, dpclip_dtype dtype, bool with_copies) {
    if (!layers || L <= 0 || L > 256 || B <= 0) return kHeaderBytes;
    dpclip_layer dense[256];
    for (int l = 0; l < L; ++l) {
        if (layers[l].kind == DPCLIP_KIND_DENSE) dense[l] = layers[l].layer;
        else memset(&dense[l], 0, sizeof(dense[l]));
    }
    size_t ws = model_scratch_bytes(layers, dense, L, B, dtype);
    const size_t staged = staged_workspace_bytes(dense, layers, L, B, dtype, with_copies);
    if (staged > ws) ws = staged;
    if (with_copies && ew_rows_total(layers, L, B) > 0) ws = round_up(ws, 256) + ew_rows_total(layers, L, B);
    return ws;
}

size_t dpclip_model_workspace_bytes(const dpclip_model_layer* layers, int L, int B, dpclip_dtype dtype) {
    return model_workspace_bytes(layers, L, B, dtype, true);
}
size_t dpclip_model_side_workspace_bytes(const dpclip_model_layer* layers, int L, int B, dpclip_dtype dtype) {
    return model_workspace_bytes(layers, L, B, dtype, false);
}

int dpclip_model_step(const dpclip_model_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                      unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                      float* norms, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = step_args_ok(layers, L, B, dtype, C, sigma, sq_layers, clip);
    if (rc) return rc;
    Lanes lanes;
    one_lane(lanes, workspace, workspace_bytes, stream);
    return step_model(layers, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes);
}

int dpclip_model_step_streams(const dpclip_model_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                              unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                              float* norms, int n_streams, void* const* streams, void* const* workspaces,
                              size_t workspace_bytes) {
    int rc = step_args_ok(layers, L, B, dtype, C, sigma, sq_layers, clip);
    if (rc) return rc;
    Lanes lanes;
    if ((rc = many_lanes(lanes, n_streams, streams, workspaces, nullptr, workspace_bytes))) return rc;
    return step_model(layers, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes);
}

int dpclip_model_step_lanes(const dpclip_model_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                              unsigned long long seed, unsigned long long stream_id0, float* sq_layers, float* clip,
                              float* norms, int n_streams, void* const* streams, void* const* workspaces,
                              const size_t* workspace_bytes) {
    if (!workspace_bytes) return DPCLIP_ERR_INVALID_ARG;
    int rc = step_args_ok(layers, L, B, dtype, C, sigma, sq_layers, clip);
    if (rc) return rc;
    Lanes lanes;
    if ((rc = many_lanes(lanes, n_streams, streams, workspaces, workspace_bytes, 0))) return rc;
    return step_model(layers, L, B, dtype, C, sigma, seed, stream_id0, sq_layers, clip, norms, lanes);
}

size_t dpclip_step_host_arena_bytes(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype) {
    if (!layers || L <= 0 || B <= 0) return 0;
    const size_t es = elt_size(dtype);
    size_t ws = dpclip_step_workspace_bytes(layers, L, B, dtype), total = 0;
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        total += round_up((size_t)B * y.T * y.d_in * es, 256);
        total += round_up((size_t)B * y.T * y.d_out * es, 256);
        total += round_up((size_t)y.d_out * y.d_in * 4, 256);
        total += round_up((size_t)y.d_out * 4, 256);
    }
    total += round_up(ws, 256);
    total += round_up((size_t)L * B * 4, 256) + 2 * round_up((size_t)B * 4, 256);
    return total;
}

int dpclip_step_host(const dpclip_layer* layers, int L, int B, dpclip_dtype dtype, float C, float sigma,
                     unsigned long long seed, unsigned long long stream_id0, float* host_clip,
                     float* host_norms, void* arena, size_t arena_bytes, void* stream) {
    if (!layers || L <= 0 || L > 64 || B <= 0 || !arena) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(arena, 256)) return DPCLIP_ERR_MISALIGNED;
    if (arena_bytes < dpclip_step_host_arena_bytes(layers, L, B, dtype)) return DPCLIP_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t es = elt_size(dtype);
    char* cur = static_cast<char*>(arena);
    auto take = [&](size_t bytes) { char* p = cur; cur += round_up(bytes, 256); return (void*)p; };

    const size_t ws_bytes = dpclip_step_workspace_bytes(layers, L, B, dtype);
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        if (y.lda != y.d_in || y.ldz != y.d_out || y.ldg != y.d_in) return DPCLIP_ERR_INVALID_ARG;
        if (!y.A || !y.Zbar || !y.gW || (y.has_bias && !y.gb)) return DPCLIP_ERR_INVALID_ARG;
    }
    void* ws = take(ws_bytes);
    float* sq = (float*)take((size_t)L * B * 4);
    if (dpclip_workspace_init(ws, ws_bytes, stream)) return DPCLIP_ERR_CUDA;

    // Arena: [workspace][sq][A_0][Zb_0][A_1][Zb_1]...[gW_0][gb_0][gW_1]...[clip][norms], every tensor on
    // the next 256-byte boundary.  When the host tensors of a direction sit back to back in the same
    // order with the same padding (one pinned buffer carved up this way), that direction is ONE copy.
    dpclip_layer dev[64];
    char* in_begin = cur;
    bool in_packed = true;
    const char* h_in0 = static_cast<const char*>(layers[0].A);
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        dev[l] = y;
        const size_t a_bytes = (size_t)B * y.T * y.d_in * es, z_bytes = (size_t)B * y.T * y.d_out * es;
        dev[l].A = take(a_bytes);
        dev[l].Zbar = take(z_bytes);
        in_packed = in_packed && static_cast<const char*>(y.A) - h_in0 == static_cast<const char*>(dev[l].A) - in_begin &&
                    static_cast<const char*>(y.Zbar) - h_in0 == static_cast<const char*>(dev[l].Zbar) - in_begin;
    }
    // a merged copy ends where the last tensor really ends: the host buffer need not extend to the padded end
    const size_t in_bytes = (size_t)(static_cast<const char*>(dev[L - 1].Zbar) - in_begin) +
                            (size_t)B * layers[L - 1].T * layers[L - 1].d_out * es;
    char* out_begin = cur;
    bool out_packed = true;
    const char* h_out0 = reinterpret_cast<const char*>(layers[0].gW);
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        dev[l].gW = (float*)take((size_t)y.d_out * y.d_in * 4);
        dev[l].gb = (float*)take((size_t)y.d_out * 4);
        out_packed = out_packed && reinterpret_cast<const char*>(y.gW) - h_out0 == reinterpret_cast<const char*>(dev[l].gW) - out_begin &&
                     (!y.has_bias || reinterpret_cast<const char*>(y.gb) - h_out0 == reinterpret_cast<const char*>(dev[l].gb) - out_begin);
        if (!y.has_bias) dev[l].gb = nullptr;
    }
    float* clip = (float*)take((size_t)B * 4);
    float* norms = (float*)take((size_t)B * 4);
    out_packed = out_packed && host_clip && host_norms &&
                 reinterpret_cast<const char*>(host_clip) - h_out0 == reinterpret_cast<const char*>(clip) - out_begin &&
                 reinterpret_cast<const char*>(host_norms) - h_out0 == reinterpret_cast<const char*>(norms) - out_begin;
    const size_t out_bytes = (size_t)(reinterpret_cast<const char*>(norms) - out_begin) + (size_t)B * 4;

    if (in_packed) {
        if (cudaMemcpyAsync(in_begin, h_in0, in_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return DPCLIP_ERR_CUDA;
    } else {
        for (int l = 0; l < L; ++l) {
            const dpclip_layer& y = layers[l];
            const size_t a_bytes = (size_t)B * y.T * y.d_in * es, z_bytes = (size_t)B * y.T * y.d_out * es;
            if (cudaMemcpyAsync(const_cast<void*>(dev[l].A), y.A, a_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess ||
                cudaMemcpyAsync(const_cast<void*>(dev[l].Zbar), y.Zbar, z_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess)
                return DPCLIP_ERR_CUDA;
        }
    }
    int rc = dpclip_step(dev, L, B, dtype, C, sigma, seed, stream_id0, sq, clip, norms, ws, ws_bytes, stream);
    if (rc) return rc;
    if (out_packed) {
        if (cudaMemcpyAsync(const_cast<char*>(h_out0), out_begin, out_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return DPCLIP_ERR_CUDA;
        return DPCLIP_OK;
    }
    for (int l = 0; l < L; ++l) {
        const dpclip_layer& y = layers[l];
        if (cudaMemcpyAsync(y.gW, dev[l].gW, (size_t)y.d_out * y.d_in * 4, cudaMemcpyDeviceToHost, st) !=
            cudaSuccess) return DPCLIP_ERR_CUDA;
        if (y.has_bias &&
            cudaMemcpyAsync(y.gb, dev[l].gb, (size_t)y.d_out * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return DPCLIP_ERR_CUDA;
    }
    if (host_clip && cudaMemcpyAsync(host_clip, clip, (size_t)B * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return DPCLIP_ERR_CUDA;
    if (host_norms && cudaMemcpyAsync(host_norms, norms, (size_t)B * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return DPCLIP_ERR_CUDA;
    return DPCLIP_OK;
}


// ---------------------------------------------------------------------------
// Clipped sum without a caller-provided workspace.
//
// Some callers have no way to hand this library device memory: a plug-in that runs inside a host
// application which owns every byte of the GPU, a service whose memory pool is carved up once at
// start-up, or code that is already inside a region where cudaMalloc is not permitted.  For them
// the split-row scratch of dpclip_clipped_grad lives in the fixed array below instead.  The array
// is part of the loaded library image: every GPU that loads libdpclip holds these 16 MB (+ 256 bytes)
// until the process exits, whether or not this entry point is ever called.
// ---------------------------------------------------------------------------
constexpr size_t kStaticScratchBytes = (size_t)16 << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kHeaderBytes + kStaticScratchBytes];

// In host code `g_static_scratch` is only a handle for the runtime, not a device address, so the
// address is looked up once per device (with that device current) and remembered.
static void* static_scratch_for_current_device(int* rc) {
    // two host threads may make the first call on a device at once: both look the same address up,
    // and the slot is published with an atomic store
    static std::atomic<void*> cached[64];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { *rc = DPCLIP_ERR_CUDA; return nullptr; }
    void* ptr = cached[dev].load(std::memory_order_acquire);
    if (!ptr) {
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) { *rc = DPCLIP_ERR_CUDA; return nullptr; }
        cached[dev].store(ptr, std::memory_order_release);
    }
    *rc = DPCLIP_OK;
    return ptr;
}

size_t dpclip_noalloc_max_output_bytes(void) { return kStaticScratchBytes / 2; }

int dpclip_clipped_grad_noalloc(const void* A, long lda, const void* Zbar, long ldz, int B, int T, int d_in,
                                int d_out, dpclip_dtype dtype, const float* clip, float* gW, long ldg, float* gb,
                                void* stream) {
    int rc = check_layer_args(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype);
    if (rc) return rc;
    if (!gW || ldg < d_in) return DPCLIP_ERR_INVALID_ARG;
    if (!aligned_to(gW, 4) || (gb && !aligned_to(gb, 4))) return DPCLIP_ERR_MISALIGNED;
    // The output, padded to 256 x 256 tiles, may take at most half of the array: room for one partial tile per
    // output tile and about as many again for the row split, which is clamped to what the array holds (at the
    // limit: 16 tiles of 512 x 256, 31 partial tiles, so 15 pairs of SMs instead of 74 -- correct, slower).
    const size_t padded = (size_t)ceil_div(d_out, 256) * 256 * ((size_t)ceil_div(d_in, 256) * 256) * 4;
    if (padded > dpclip_noalloc_max_output_bytes()) return DPCLIP_ERR_WORKSPACE;
    void* scratch = static_scratch_for_current_device(&rc);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    // the array keeps whatever the previous call left: the status header has to start at zero (the
    // partial tiles need no clearing, every tile that is read is written first)
    if (cudaMemsetAsync(scratch, 0, kHeaderBytes, st) != cudaSuccess) return DPCLIP_ERR_CUDA;
    if (tc_eligible(A, lda, Zbar, ldz, dtype))
        return launch_zta_tc(A, lda, Zbar, ldz, B, T, d_in, d_out, false, 0, clip, gW, ldg, gb, nullptr, scratch,
                             kHeaderBytes + kStaticScratchBytes, nullptr, nullptr, st, /*fit_to_workspace=*/true);
    return launch_simt_grad(A, lda, Zbar, ldz, B, T, d_in, d_out, dtype, clip, gW, ldg, gb, st);
}

}  // extern "C"
