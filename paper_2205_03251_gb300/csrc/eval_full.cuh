// Full interpretation of a population (Sec. 4.2), split at the cached
// skeleton: first every small subtree hanging off a cached node (in
// parallel, one warp per subtree and case block), then the cached nodes
// bottom up, then the fitness of each root.
#pragma once
#include "fused.cuh"

// Work item of entry e: the part of its subtree not covered by large
// children -- the whole subtree when both children are small, else the
// small child (its value is parked in e's slot until the skeleton pass).
__global__ void k_build_items(DevPop d, const uint32_t* __restrict__ e_tree) {
    if (halted(d)) return;
    const uint32_t ne = d.e_off[d.P];
    if (ne > d.Ecap) return;
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += gridDim.x * blockDim.x) {
        const int32_t c0 = d.e_c0[e], c1 = d.e_c1[e];
        uint32_t s = 0, len = 0;
        if (c0 < 0 && c1 < 0) { s = d.e_pos[e]; len = d.e_end[e] - s; }
        else if (c0 >= 0 && c1 < 0) { s = d.e_end[c0]; len = d.e_end[e] - s; }
        else if (c0 < 0 && c1 >= 0) { s = d.e_pos[e] + 1; len = d.e_pos[c1] - s; }
        const uint32_t buf = d.buf[e_tree[e]];
        d.it_desc[e] = make_uint4(s, len, d.e_slot[e], buf);
        const uint32_t op = d.arena[(size_t)buf * d.cap + d.e_pos[e]];
        const uint32_t oslot = (c0 >= 0 && c1 >= 0) ? d.e_slot[c1] : d.e_slot[e];
        d.sk_desc[e] = make_uint4(d.e_slot[e], oslot, op | ((c0 >= 0) ? 0x100u : 0u) | ((c1 >= 0) ? 0x200u : 0u),
                                  (uint32_t)c1);
        d.order[e] = e;
    }
}

// Shared memory of a k_eval_items CTA: the leaf table (first, so that its
// addresses fit 16 bits), then per warp a stack window and the instruction
// list of one chunk.
template <int K, int V>
struct ItemsLayout {
    __host__ __device__ static size_t warp_bytes(int W) { return SmemLayout<K>::stack_bytes(W) + FX_CODE_BYTES; }
    __host__ __device__ static size_t total(int W, uint32_t ncb) {
        return FxTable<K, V>::bytes(ncb) + GP_WARPS * warp_bytes(W);
    }
};

// Persistent warps over (item, case block) units.  The next unit's index,
// descriptor and first words are fetched while the current one is evaluated.
// Bound by the indirect branch of each instruction (about 24 cycles of an
// SM quarter, whatever it branches to; 0.53 instructions a node on grafted
// trees), which 16 warps per SM saturate.  500 grafted trees of ~1e6 nodes x
// 48 cases: 14.4 ms node by node, 6.6 ms now; 2,001 uneven integer trees 1.59
// -> 0.95 ms; 600 uneven trees x 1,000 cases 5.57 -> 3.2 ms.  The words are
// read straight from the tree, a chunk ahead (no staged copy).
template <int K, int V>
__global__ void __launch_bounds__(GP_WARPS * 32, K == 4 ? 3 : V == VF ? 4 : 5) k_eval_items(DevPop d) {
    if (halted(d)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    FxTable<K, V>::fill(reinterpret_cast<float*>(smem_raw), d.consts, d.ncb);
    __syncthreads();
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t wb = sm + FxTable<K, V>::bytes(d.ncb) + warp * (uint32_t)ItemsLayout<K, V>::warp_bytes((int)d.W);
    FxCtx<K> c;
    c.stack = wb + lane * K * 4;
    c.code = wb + (uint32_t)SmemLayout<K>::stack_bytes((int)d.W);
    c.lo = lane * K * 4;
    c.W = d.W;
    c.maxd = d.maxdepth;
    const uint32_t gwarp = blockIdx.x * GP_WARPS + warp;
    c.g = d.ovf + (size_t)gwarp * d.maxdepth * 32 * K;
    const uint32_t ne = d.e_off[d.P];
    if (ne > d.Ecap) return;
    const uint32_t nunits = ne * d.ncb;
    unsigned long long ops_done = 0;     // nodes interpreted (once per item, not per case block)

    // Three units are under way in a warp: the one being evaluated, the next
    // one's first words in flight, and the descriptor of the one after it.
    // The first unit of each warp is its own (spread over the CTAs, so that a
    // small population uses every SM), the others come from the queue.
    const uint32_t nwarps = gridDim.x * GP_WARPS;
    uint32_t qnext = 0;                                  // lane 0: a unit taken from the queue ahead
    if (lane == 0) qnext = nwarps + atomicAdd(&d.q[Q_ITEMS], 1u);
    auto unit = [&]() -> uint32_t {
        const uint32_t u = __shfl_sync(FULL, qnext, 0);
        if (lane == 0 && u < nunits) qnext = nwarps + atomicAdd(&d.q[Q_ITEMS], 1u);
        return u;
    };
    // a descriptor under way is one register: lane k holds word k
    auto fetch = [&](uint32_t u) -> uint32_t {
        return (u < nunits && lane < 4) ? reinterpret_cast<const uint32_t*>(d.it_desc)[4 * (size_t)(u / d.ncb) + lane] : 0u;
    };
    auto words = [&](uint32_t t, uint32_t& a0, uint32_t& a1) {
        const uint32_t s = __shfl_sync(FULL, t, 0), len = __shfl_sync(FULL, t, 1), buf = __shfl_sync(FULL, t, 3);
        a0 = a1 = 0xFFFFFFFFu;
        if (len) {
            const uint32_t* tree = reinterpret_cast<const uint32_t*>(d.arena + (size_t)buf * d.cap);
            fx_first([&](uint32_t q) { return __ldg(tree + (q >> 2)); }, s, s + len, a0, a1);
        }
    };
    uint32_t u0 = warp * gridDim.x + blockIdx.x, w0, w1;
    uint32_t t0 = fetch(u0);
    uint32_t u1 = unit(), t1 = fetch(u1);
    words(t0, w0, w1);
    while (u0 < nunits) {
        uint32_t v0, v1;
        words(t1, v0, v1);
        const uint32_t u2 = unit();
        const uint32_t t2 = fetch(u2);
        const uint32_t s = __shfl_sync(FULL, t0, 0), len = __shfl_sync(FULL, t0, 1);
        if (len) {
            const uint32_t cbk = u0 % d.ncb;
            load_cases<K>(d, cbk, c.x);
            c.lt = FxTable<K, V>::at(sm, cbk);
            const uint32_t* tree = reinterpret_cast<const uint32_t*>(d.arena + (size_t)__shfl_sync(FULL, t0, 3) * d.cap);
            float a[K];
            const bool ok = fx_run<K, V>([&](uint32_t q) { return __ldg(tree + (q >> 2)); }, s, s + len, w0, w1, c, a);
            if (!ok && lane == 0) set_status(d.status, ST_STACK);
            store_slot<K>(d, __shfl_sync(FULL, t0, 2), cbk, a);
            if (cbk == 0) ops_done += len;
        }
        u0 = u1; t0 = t1; w0 = v0; w1 = v1;
        u1 = u2; t1 = t2;
    }
    if (lane == 0 && ops_done) { atomicAdd(&d.acc_ops[0], ops_done); atomicAdd(&d.acc_ops[2], ops_done); }
}

// Cached nodes bottom up: entries of a tree in decreasing position order,
// so both children of a node are done before it.  A node with one large
// child has that child at the next entry index (no other cached node lies
// between them), a node with two has its left child there.  Entries are
// taken in groups of SKB: descriptors (prefetched one group ahead) and
// operand vectors are loaded first -- they do not depend on the running
// value -- then combined in order; a right child inside the same group is
// taken from the group's own results.
#define SKB 16
template <int K, int V>
__global__ void __launch_bounds__(GP_WARPS * 32) k_eval_skeleton(DevPop d) {
    if (halted(d)) return;
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    const int lane = lane_id();
    if (d.e_off[d.P] > d.Ecap) return;
    for (uint32_t tree = gw; tree < d.P; tree += nw) {
        const uint32_t e0 = d.e_off[tree], e1 = d.e_off[tree + 1];
        unsigned long long cnt = 0;
        for (uint32_t cbk = 0; cbk < d.ncb; ++cbk) {
            float prev[K];
#pragma unroll
            for (int k = 0; k < K; ++k) prev[k] = 0.f;
            uint4 md = make_uint4(0, 0, 0, 0);
            if (e1 > e0 && lane < SKB && (uint32_t)lane < e1 - e0) md = d.sk_desc[e1 - 1 - lane];
            for (uint32_t top = e1; top > e0;) {
                const uint32_t nb = (top - e0 < SKB) ? top - e0 : SKB;
                const uint32_t ntop = top - nb;
                uint4 mdn = make_uint4(0, 0, 0, 0);
                if (ntop > e0 && lane < SKB && (uint32_t)lane < ntop - e0) mdn = d.sk_desc[ntop - 1 - lane];
                float opnd[SKB][K];
                uint32_t slots[SKB], info[SKB], c1s[SKB];
#pragma unroll
                for (int j = 0; j < SKB; ++j) {
                    slots[j] = __shfl_sync(FULL, md.x, j);
                    const uint32_t os = __shfl_sync(FULL, md.y, j);
                    info[j] = __shfl_sync(FULL, md.z, j);
                    c1s[j] = __shfl_sync(FULL, md.w, j);
                    if (j < (int)nb) load_slot<K>(d, os, cbk, opnd[j]);
                }
                float done[SKB][K];
#pragma unroll
                for (int j = 0; j < SKB; ++j) {
                    if (j < (int)nb) {
                        const bool has0 = info[j] & 0x100u, has1 = info[j] & 0x200u;
                        const uint32_t op = info[j] & 0xFFu;
                        float val[K];
                        if (!has0 && !has1) {
#pragma unroll
                            for (int k = 0; k < K; ++k) val[k] = opnd[j][k];
                        } else {
                            float o[K];
#pragma unroll
                            for (int k = 0; k < K; ++k) o[k] = opnd[j][k];
                            if (has0 && has1) {
#pragma unroll
                                for (int jj = 0; jj < j; ++jj)
                                    if (c1s[j] == top - 1 - jj) {
#pragma unroll
                                        for (int k = 0; k < K; ++k) o[k] = done[jj][k];
                                    }
                            }
                            if (has0) {                       // left = entry e+1 = prev
#pragma unroll
                                for (int k = 0; k < K; ++k) val[k] = prev[k];
                                apply_vec<K, V>(op, val, o);
                            } else {                          // right = entry e+1 = prev
#pragma unroll
                                for (int k = 0; k < K; ++k) val[k] = o[k];
                                apply_vec<K, V>(op, val, prev);
                            }
                            store_slot<K>(d, slots[j], cbk, val);
                            if (cbk == 0) ++cnt;
                        }
#pragma unroll
                        for (int k = 0; k < K; ++k) { done[j][k] = val[k]; prev[k] = val[k]; }
                    }
                }
                top = ntop;
                md = mdn;
            }
        }
        if (lane == 0 && cnt) atomicAdd(&d.acc_ops[0], cnt);
    }
}

// Fitness of every tree from its root's cached vector (a warp per tree).
__global__ void k_fitness(DevPop d) {
    if (halted(d)) return;
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    if (d.e_off[d.P] > d.Ecap) return;
    for (uint32_t tree = gw; tree < d.P; tree += nw) {
        const float* v = d.slots + (size_t)d.e_slot[d.e_off[tree]] * d.Cpad;
        const float f = fitness_warp(d, [&](uint32_t j) { return __ldcg(v + j); });
        if (lane_id() == 0) {
            d.fit[tree] = f;
            atomicAdd(&d.acc_ops[1], (unsigned long long)d.size[tree]);
        }
    }
}
