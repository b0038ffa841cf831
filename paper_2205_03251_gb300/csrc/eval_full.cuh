// Full interpretation of a population (Sec. 4.2), split at the cached
// skeleton: first every small subtree hanging off a cached node (in
// parallel, one warp per subtree and case block), then the cached nodes
// bottom up, then the fitness of each root.
#pragma once
#include "fused.cuh"

// Entries a warp of the skeleton pass evaluates by itself before it climbs.
// (32: bushy trees climb a twentieth of their entries; with four cases per lane shared memory
// for the values of 8.)
__host__ __device__ constexpr uint32_t sk_group(uint32_t K) { return K == 4 ? 8u : 32u; }
// Does entry e's cached subtree (its entries are contiguous) fit a group?
__device__ __forceinline__ bool sk_small(const DevPop& d, const uint32_t* __restrict__ e_tree, uint32_t e) {
    const uint32_t x = e + sk_group(d.K);
    return x >= d.e_off[e_tree[e] + 1] || d.e_pos[x] >= d.e_end[e];
}

// Work item of entry e: the part of its subtree not covered by large
// children -- the whole subtree when both children are small, else the
// small child (its value is parked in e's slot until the skeleton pass).
// Also the list of entries the skeleton pass starts from (d.order).
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
        // the climbs of the skeleton pass start at the largest entries whose cached subtree is small
        d.e_flag[e] = 0u;
        const int32_t p = d.e_par[e];
        const uint32_t here = __activemask();
        const bool start = sk_small(d, e_tree, e) && (p < 0 || !sk_small(d, e_tree, (uint32_t)p));
        const uint32_t mk = __ballot_sync(here, start);
        if (start) {
            const int lead = __ffs(mk) - 1;
            uint32_t at = 0;
            if (lane_id() == lead) at = atomicAdd(&d.q[Q_SKEL], (uint32_t)__popc(mk));
            at = __shfl_sync(mk, at, lead);
            d.order[at + __popc(mk & ((1u << lane_id()) - 1u))] = e;
        }
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
// Grafted trees: bound by the indirect branch of each instruction (about 24
// cycles of an SM quarter, whatever it branches to; 0.53 instructions a node),
// which 16 warps per SM saturate.  Uneven trees: bound by the units -- half of
// their items are one leaf, 94 % fit a chunk, and each costs a place in the
// queue, a descriptor, a decode and a value vector whatever its length.  500
// grafted trees of ~1e6 nodes x 48 cases: 12.6 ms node by node, 6.7 ms now;
// 2,001 uneven integer trees 1.57 -> 0.94 ms; 600 uneven trees x 1,000 cases
// 4.98 -> 2.13 ms.  The words are read straight from the tree, a chunk ahead
// (no staged copy).
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

// Cached nodes bottom up.  A warp (per case block) first evaluates a whole
// small cached subtree, up to sk_group entries, from its last entry to its
// first: a node's left or only cached child is the next entry, whose value is
// the running one, its right one was computed earlier and waits in shared
// memory, and the items' values it combines with depend on nothing, so they
// are loaded SKB at a time.  Then it climbs.  The run of nodes with one cached
// child above an entry is a run of descending indexes: their descriptors come
// in one load of 32.  At a node with two cached children the warp that
// arrives first leaves its value in the slot and ends; the second one
// combines both and goes on (a bit per node and case block, set by atomicOr).
// No warp waits.  Bound by latency along a tree's longest chain; every chain
// and case block runs at once, where a warp per tree took the chains and the
// case blocks one after another: 500 grafted trees of ~1e6 nodes x 48 cases
// 1.03 -> 0.32 ms, 1,500 uneven trees over the 11-multiplexer 1.16 -> 0.44 ms,
// 600 uneven trees x 1,000 cases 13.4 -> 0.51 ms.  cb0, ncbp: the case blocks
// of this launch (at most 32, the bits of a flag word).
#define SKB 8
#define SK_WARPS 4
template <int K, int V>
__global__ void __launch_bounds__(SK_WARPS * 32) k_eval_skeleton(DevPop d, uint32_t cb0, uint32_t ncbp) {
    if (halted(d)) return;
    __shared__ __align__(16) float done[SK_WARPS][sk_group(K)][32 * K];           // values of the group's entries
    const int lane = lane_id();
    const uint32_t ne = d.e_off[d.P];
    if (ne > d.Ecap) return;
    const uint32_t nunits = d.q[Q_SKEL] * ncbp, nwarps = gridDim.x * SK_WARPS;
    float (*mine)[32 * K] = done[threadIdx.x >> 5];
    uint32_t cnt = 0;
    // Units from a queue, each taken when the warp is free: a unit taken ahead
    // would be held up by the climb before it, and every unit above would wait.
    uint32_t u = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    while (u < nunits) {
        const uint32_t cb = u % ncbp, cbk = cb0 + cb;
        uint32_t e = d.order[u / ncbp];
        float val[K];
        uint4 gd = make_uint4(0, 0, 0, 0);
        uint32_t pos = 0xFFFFFFFFu, tree = 0;
        const uint32_t x = e + lane, end = d.e_end[e];
        if (lane < (int)sk_group(K) && x < ne) { gd = d.sk_desc[x]; pos = d.e_pos[x]; tree = d.e_tree[x]; }
        const uint32_t own = __shfl_sync(FULL, tree, 0);
        const uint32_t n = __popc(__ballot_sync(FULL, pos < end && tree == own));
        uint4 md = make_uint4(0, 0, 0, 0);                                   // the entries below e: lane l has e - 1 - l
        if ((uint32_t)lane < e) md = d.sk_desc[e - 1 - lane];
#pragma unroll
        for (int k = 0; k < K; ++k) val[k] = 0.f;
        for (int top = (int)n; top > 0; top -= SKB) {
            float opnd[SKB][K];
#pragma unroll
            for (int j = 0; j < SKB; ++j) {
                const uint32_t os = __shfl_sync(FULL, gd.y, top - 1 - j);
                const uint32_t info = __shfl_sync(FULL, gd.z, top - 1 - j);
                if (top - 1 - j >= 0 && (info & 0x300u) != 0x300u) load_slot<K>(d, os, cbk, opnd[j]);
            }
#pragma unroll
            for (int j = 0; j < SKB; ++j) {
                const int l = top - 1 - j;
                const uint32_t info = __shfl_sync(FULL, gd.z, l), slot = __shfl_sync(FULL, gd.x, l);
                const uint32_t right = __shfl_sync(FULL, gd.w, l) - e;
                if (l >= 0) {
                    if ((info & 0x300u) == 0u) {                             // an item's value
#pragma unroll
                        for (int k = 0; k < K; ++k) val[k] = opnd[j][k];
                    } else {
                        if ((info & 0x300u) == 0x300u) vload<K>(&mine[right][lane * K], opnd[j]);
                        else if (!(info & 0x100u)) {                         // the running value is the right operand
#pragma unroll
                            for (int k = 0; k < K; ++k) { const float t = val[k]; val[k] = opnd[j][k]; opnd[j][k] = t; }
                        }
                        apply_vec<K, V>(info & 0xFFu, val, opnd[j]);
                        store_slot<K>(d, slot, cbk, val);
                        if (cbk == 0) ++cnt;
                    }
                    vstore<K>(&mine[l][lane * K], val);
                }
            }
        }
        for (;;) {
            // the run of nodes with one cached child above e
            const bool h0 = md.z & 0x100u, h1 = md.z & 0x200u;
            const uint32_t other = __ballot_sync(FULL, h0 == h1);            // none or two: the run ends
            const uint32_t run = other ? (uint32_t)__ffs(other) - 1u : 32u;
            const int32_t up = run < 32u ? d.e_par[e - run] : 0;             // (needed after the run)
            // A long run (a chain of a deep tree) takes its operands SKB at a time and its descriptors 32 at a time: what
            // comes after the first group is fetched towards the L2 meanwhile.  (100 combs of up to 60,000 nodes, integers:
            // 9.3 ms a tree per warp and 16 at a time, 10.4 in climbs, 7.9 with this; the 11-multiplexer 6.3, 7.0, 5.7.)
            if (run > SKB) {
                const float* p = d.slots + (size_t)md.y * d.Cpad + cbk * 32 * K;
                if ((uint32_t)lane >= SKB && (uint32_t)lane < run) {
#pragma unroll
                    for (int k = 0; k < K; ++k) prefetch_l2(p + 32 * k);
                }
                if (run == 32 && e >= 33u + (uint32_t)lane) prefetch_l2(d.sk_desc + (e - 33u - lane));
            }
            for (uint32_t j0 = 0; j0 < run; j0 += SKB) {
                float opnd[SKB][K];
#pragma unroll
                for (int j = 0; j < SKB; ++j) {
                    const uint32_t os = __shfl_sync(FULL, md.y, (int)j0 + j);
                    if (j0 + j < run) load_slot<K>(d, os, cbk, opnd[j]);
                }
#pragma unroll
                for (int j = 0; j < SKB; ++j) {
                    const uint32_t info = __shfl_sync(FULL, md.z, (int)j0 + j), slot = __shfl_sync(FULL, md.x, (int)j0 + j);
                    if (j0 + j < run) {
                        if (!(info & 0x100u)) {                              // the running value is the right operand
#pragma unroll
                            for (int k = 0; k < K; ++k) { const float t = val[k]; val[k] = opnd[j][k]; opnd[j][k] = t; }
                        }
                        apply_vec<K, V>(info & 0xFFu, val, opnd[j]);
                        store_slot<K>(d, slot, cbk, val);
                    }
                }
            }
            e -= run;
            if (cbk == 0) cnt += run;                       // nodes combined, once
            if (run == 32) {
                md = make_uint4(0, 0, 0, 0);
                if ((uint32_t)lane < e) md = d.sk_desc[e - 1 - lane];
                continue;
            }
            // e's parent has two cached children (e the left one when it is the entry before e), or e is a root
            const uint32_t below = __shfl_sync(FULL, md.z, (int)run);
            const bool left = (below & 0x300u) == 0x300u;
            const int32_t p = left ? (int32_t)e - 1 : up;
            if (p < 0) break;
            // all that the second to arrive needs but the value, loaded before it is known who that is
            const uint32_t info = left ? below : d.sk_desc[p].z;
            const uint32_t slot = left ? __shfl_sync(FULL, md.x, (int)run) : d.sk_desc[p].x;
            const uint32_t sib = left ? __shfl_sync(FULL, md.y, (int)run) : d.sk_desc[p + 1].x;
            md = make_uint4(0, 0, 0, 0);
            if (lane < p) md = d.sk_desc[p - 1 - lane];
            uint32_t first = 0;
            __threadfence();
            __syncwarp();
            if (lane == 0) first = !(atomicOr(&d.e_flag[p], 1u << cb) & (1u << cb));
            if (__shfl_sync(FULL, first, 0)) break;
            __threadfence();
            float o[K];
            load_slot<K>(d, sib, cbk, o);
            if (!left) {
#pragma unroll
                for (int k = 0; k < K; ++k) { const float t = val[k]; val[k] = o[k]; o[k] = t; }
            }
            apply_vec<K, V>(info & 0xFFu, val, o);
            store_slot<K>(d, slot, cbk, val);
            e = (uint32_t)p;
            if (cbk == 0) ++cnt;
        }
        __syncwarp();
        if (lane == 0) u = nwarps + atomicAdd(&d.q[Q_CLIMB], 1u);
        u = __shfl_sync(FULL, u, 0);
    }
    if (lane == 0 && cnt) atomicAdd(&d.acc_ops[0], (unsigned long long)cnt);
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
