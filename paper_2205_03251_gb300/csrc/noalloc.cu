// gp_eval_small_noalloc: full evaluation of a batch of small trees with no
// device allocation at all.
//
// Some callers cannot call cudaMalloc: a plug-in whose host process has
// handed the whole device memory to its own pool allocator (a cudaMalloc
// there fails, or fragments memory the host accounts for), a real-time loop
// that must not take the implicit device synchronisation an allocation can
// bring, or an embedding whose memory is fixed at start-up.  They still own
// their inputs and outputs, so this entry point takes device pointers to
// both and keeps the only scratch it needs -- the interpreter's deep-stack
// overflow area, a work counter and a status word -- in one file-scope
// device array of fixed size, loaded with the library and held by every GPU
// that loads it until the process exits.
//
// The scratch array is shared by every call on a device and keeps the
// previous call's contents; each call clears the counter and status it needs
// before launching.  Two calls whose work overlaps on the GPU (different
// streams, or one not yet finished when the next is issued on another
// stream) race on that array and give undefined results: serialise them.
// Each call synchronises its stream before it returns, to read the status.
#include "gpfdp.h"

#include <cstdint>
#include <mutex>

#include "common.cuh"
#include "fused.cuh"

namespace {

constexpr int NA_MAX_NODES = 1023;            // largest tree: at most 512 leaves, so the stack
constexpr int NA_MAXD = 520;                  //   never holds more than 514 entries
constexpr int NA_WARPS = 16;                  // warps per CTA, a CTA per SM: what the interpreter's branches need
constexpr int NA_WIN_FLOATS = 96 * 32;        // a warp's stack window: 96 / K entries
constexpr int NA_SLOTS = 64;                  // overflow stacks
constexpr size_t NA_OVF_FLOATS = (size_t)NA_SLOTS * NA_MAXD * 32 * 2;
// control words: 0 work counter, 1 status, 2 tickets for overflow stacks, 8 + 8 s the turn of stack s (a 32-byte sector each)
constexpr int NA_CTL = 8 + 8 * NA_SLOTS;
constexpr size_t NA_SCRATCH_FLOATS = NA_OVF_FLOATS + NA_CTL;   // overflow stacks, then control words
constexpr uint32_t NA_SPIN = 1u << 22;        // bound on the polls for a stack between two of its turns
}  // namespace

// The scratch: 64 overflow stacks (8.5 MB: 520 entries x 32 lanes x 2 cases x
// 4 bytes each) and the control words.  Any warp may run; one whose tree is
// deeper than its window in shared memory takes an overflow stack until that
// tree is done.
static __device__ __align__(256) float g_noalloc_scratch[NA_SCRATCH_FLOATS];

namespace {

struct NaArgs {
    const uint8_t* ops;
    size_t ops_bytes;
    const uint64_t* off;
    uint32_t n_trees;
    const float* x;
    const float* t;
    const float* consts;
    uint32_t n_cases;
    float* values;
    float* fitness;
    float* scratch;       // device address of g_noalloc_scratch
};

template <int K>
struct NaLayout {
    static constexpr uint32_t table = FxTable<K, VF>::row * 256;
    static constexpr uint32_t warp_bytes = NA_WIN_FLOATS * 4 + FX_CODE_BYTES;
    static constexpr uint32_t total = table + NA_WARPS * warp_bytes;
};

// A warp per tree (all of its case blocks in turn: the fitness sums them in
// case order), or, when there are fewer trees than CTAs, a CTA per tree with
// its warps on the case blocks.  The first trees go round the CTAs, so that a
// few trees run on as many SMs; the others come from the counter.  3,000
// uneven trees of up to 1,023 nodes x 100 cases: 2,150 us with 64 warps on
// the whole chip, 129 us with 16 on each SM.
template <int K>
__global__ void __launch_bounds__(NA_WARPS * 32) k_eval_small_noalloc(NaArgs a, uint32_t by_cta) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    FxTable<K, VF>::fill(reinterpret_cast<float*>(smem_raw), a.consts, 1);
    __syncthreads();
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t wb = sm + NaLayout<K>::table + warp * NaLayout<K>::warp_bytes;
    volatile uint32_t* ctl = reinterpret_cast<volatile uint32_t*>(a.scratch + NA_OVF_FLOATS);
    uint32_t* counter = const_cast<uint32_t*>(ctl);
    uint32_t* status = counter + 1;
    FxCtx<K> c;
    c.stack = wb + lane * K * 4;
    c.code = wb + NA_WIN_FLOATS * 4;
    c.lt = sm;
    c.lo = 0;
    c.W = 96 / K;
    c.maxd = NA_MAXD;
    c.g = nullptr;
    int held = -1;
    // An overflow stack: the warp with ticket t takes stack t % NA_SLOTS after
    // the t / NA_SLOTS warps before it have had it.  A holder never waits, so
    // every turn comes, in the order of the tickets; a wait may be as long as
    // the batch, but a turn lasts no longer than a tree, so the polls are
    // counted anew with each turn.  (A free stack for whoever takes it first
    // drew thousands of warps to one word, and without an order one of them
    // could miss every stack.  20,000 trees of 121 nodes and depth 61 x 100
    // cases 14.0 -> 10.7 ms.)
    auto need = [&]() -> bool {
        if (held >= 0) return true;
        int got = -1;
        if (lane == 0) {
            const uint32_t t = atomicAdd(counter + 2, 1u), mine = t / NA_SLOTS;
            const volatile uint32_t* turn = ctl + 8 + 8 * (t % NA_SLOTS);
            uint32_t idle = 0, now = *turn;
            while (now != mine && idle < NA_SPIN) {
                __nanosleep(64);
                const uint32_t was = now;
                now = *turn;
                idle = now == was ? idle + 1 : 0;
            }
            if (now == mine) got = (int)(t % NA_SLOTS);
            else atomicOr(status, 4u);
            __threadfence();
        }
        held = __shfl_sync(FULL, got, 0);
        if (held >= 0) c.g = a.scratch + (size_t)held * NA_MAXD * 32 * 2;
        return held >= 0;
    };
    auto release = [&]() {
        if (held < 0) return;
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(counter + 8 + 8 * held, 1u);
        held = -1;
    };
    const uint32_t ncb = (a.n_cases + 32 * K - 1) / (32 * K);
    const uint32_t first = by_cta ? 1u : (uint32_t)NA_WARPS;        // trees a CTA starts with
    const uint32_t* words = reinterpret_cast<const uint32_t*>(a.ops);
    uint32_t i = by_cta ? blockIdx.x : warp * gridDim.x + blockIdx.x;
    while (i < a.n_trees) {
        const uint64_t s64 = a.off[i], e64 = a.off[i + 1];
        const uint64_t n = e64 - s64;
        // ops_bytes is a multiple of 16, so e64 <= ops_bytes also keeps the
        // words read inside the buffer (no rounding that could wrap)
        const bool fits = e64 >= s64 && n != 0 && n <= NA_MAX_NODES && e64 <= a.ops_bytes;
        if (!fits && lane == 0) atomicOr(status, 1u);
        float fit = 0.0f;
        if (fits) {
            const uint32_t s = (uint32_t)(s64 & 3u), e = s + (uint32_t)n;
            const uint32_t* tree = words + (s64 >> 2);
            auto ld = [&](uint32_t q) { return __ldg(tree + (q >> 2)); };
            for (uint32_t cb = by_cta ? warp : 0; cb < ncb; cb += by_cta ? NA_WARPS : 1) {
                // lanes past the last case repeat it: their values are not written
#pragma unroll
                for (int k = 0; k < K; ++k) c.x[k] = a.x[min(cb * 32 * K + k * 32 + lane, a.n_cases - 1)];
                uint32_t w0, w1;
                fx_first(ld, s, e, w0, w1);
                float v[K];
                bool ok = fx_run<K, VF>(ld, s, e, w0, w1, c, v, need);
                if (!ok && lane == 0) atomicOr(status, 2u);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const uint32_t cc = cb * 32 * K + k * 32 + lane;
                    const bool in = cc < a.n_cases;
                    if (in) a.values[(size_t)i * a.n_cases + cc] = v[k];
                    if (!by_cta) {
                        // fitness in case order: the terms of 32 cases at once, then their sum
                        const float term = in ? fabsf(__fsub_rn(v[k], a.t[cc])) : 0.0f;
                        const uint32_t m = min(32u, a.n_cases - min(a.n_cases, cb * 32 * K + k * 32));
                        for (uint32_t l = 0; l < m; ++l) fit = __fadd_rn(fit, __shfl_sync(FULL, term, l));
                    }
                }
            }
            release();
        }
        if (by_cta) {
            __syncthreads();                        // the tree's values, all of its case blocks
            if (warp == 0 && fits)
                for (uint32_t b = 0; b < a.n_cases; b += 32) {
                    const uint32_t j = b + lane, m = min(32u, a.n_cases - b);
                    const float term = j < a.n_cases ? fabsf(__fsub_rn(a.values[(size_t)i * a.n_cases + j], a.t[j])) : 0.0f;
                    for (uint32_t l = 0; l < m; ++l) fit = __fadd_rn(fit, __shfl_sync(FULL, term, l));
                }
        }
        if (fits && lane == 0 && (!by_cta || warp == 0)) a.fitness[i] = fit;
        if (by_cta) {
            i += gridDim.x;                         // (by_cta: at most one tree per CTA)
        } else {
            uint32_t v = 0;
            if (lane == 0) v = atomicAdd(counter, 1u);
            i = gridDim.x * first + __shfl_sync(FULL, v, 0);
        }
    }
}

std::mutex g_na_mu;
// device address of the scratch per device ordinal, and the context it was
// looked up in: a context destroyed and re-created (cudaDeviceReset) loads
// the module again, so the address is looked up again in the new context
float* g_na_ptr[64] = {};
void* g_na_ctx[64] = {};
int g_na_nsm[64] = {};

// the current context through the driver entry point (no link-time
// dependency on the driver library)
typedef int (*CtxGetCurrentFn)(void**);
void* current_context() {
    static CtxGetCurrentFn fn = nullptr;
    static bool looked = false;
    if (!looked) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 4000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<CtxGetCurrentFn>(p);
        looked = true;
    }
    void* ctx = nullptr;
    if (fn && fn(&ctx) != 0) ctx = nullptr;
    return ctx;
}

}  // namespace

extern "C" int gp_eval_small_noalloc(const uint8_t* d_ops, size_t ops_bytes, const uint64_t* d_off,
                                     uint32_t n_trees, const float* d_x, const float* d_t,
                                     const float* d_consts, uint32_t n_cases, float* d_values,
                                     float* d_fitness, void* stream, uint32_t* status_out) {
    if (status_out) *status_out = 0;
    if (!d_ops || !d_off || !d_x || !d_t || !d_consts || !d_values || !d_fitness) return GP_EINVAL;
    if (n_cases == 0 || n_cases > 4096) return GP_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_ops) & 15u) || (ops_bytes & 15u)) return GP_EINVAL;
    if (n_trees == 0) return GP_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return GP_ECUDA;
    float* scratch = nullptr;
    int nsm = 0;
    {
        // set-up, once per device (and context), with that device current: the
        // host-side name of the array is not a device address, so ask the
        // runtime for it
        std::lock_guard<std::mutex> lk(g_na_mu);
        void* ctx = current_context();
        if (!g_na_ptr[dev] || !ctx || ctx != g_na_ctx[dev]) {
            void* p = nullptr;
            // (creates the device's context if it does not exist yet)
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) return GP_ECUDA;
            if (cudaFuncSetAttribute(k_eval_small_noalloc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)NaLayout<1>::total) != cudaSuccess ||
                cudaFuncSetAttribute(k_eval_small_noalloc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)NaLayout<2>::total) != cudaSuccess ||
                cudaDeviceGetAttribute(&g_na_nsm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
                return GP_ECUDA;
            g_na_ptr[dev] = static_cast<float*>(p);
            g_na_ctx[dev] = current_context();
        }
        scratch = g_na_ptr[dev];
        nsm = g_na_nsm[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the work counter, the status word, the tickets and the turns start at zero on every call
    if (cudaMemsetAsync(scratch + NA_OVF_FLOATS, 0, NA_CTL * sizeof(float), st) != cudaSuccess) return GP_ECUDA;
    NaArgs a{d_ops, ops_bytes, d_off, n_trees, d_x, d_t, d_consts, n_cases, d_values, d_fitness, scratch};
    // (four cases per lane would halve the window: most larger trees would then queue for an overflow stack, 970 us
    // instead of 133 us for 3,000 trees x 100 cases)
    const int K = n_cases <= 32 ? 1 : 2;
    const uint32_t ncb = (n_cases + 32 * K - 1) / (32 * K);
    const uint32_t by_cta = (ncb > 1 && n_trees <= (uint32_t)nsm) ? 1u : 0u;
    const uint32_t grid = n_trees < (uint32_t)nsm ? n_trees : (uint32_t)nsm;
    if (K == 1) k_eval_small_noalloc<1><<<grid, NA_WARPS * 32, NaLayout<1>::total, st>>>(a, by_cta);
    else k_eval_small_noalloc<2><<<grid, NA_WARPS * 32, NaLayout<2>::total, st>>>(a, by_cta);
    if (cudaGetLastError() != cudaSuccess) return GP_ECUDA;
    uint32_t flags = 0;
    if (cudaMemcpyAsync(&flags, scratch + NA_OVF_FLOATS + 1, sizeof flags, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return GP_ECUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return GP_ECUDA;
    if (status_out) *status_out = flags;
    if (flags & 1u) return GP_ECAPACITY;
    if (flags & 4u) return GP_ETIMEOUT;
    if (flags & 2u) return GP_EINVAL;
    return GP_OK;
}
