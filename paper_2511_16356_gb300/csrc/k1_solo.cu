// Wilson's loop-erased-walk sampler (Sec. 2.2), one walker per tree with the
// arrows drawn ahead.  The trees, step counts and parent-first orders are those
// of k1_wilson.cu: vertex u's k-th arrow is bounded(seed, u, k, sample, WALK,
// deg u), and by cycle popping neither the start order nor the walker matters.
//
// What bounds a sequential walker is the chain of one departure: load the word
// of the vertex, ten dependent Philox rounds, select the neighbour, load its
// word.  Here the word of a vertex outside the tree holds a queue of its next
// arrows as neighbour indices, so a departure is a load, a select and a shift; an
// empty queue is refilled by the warp, one arrow per lane.  The first queue of
// every vertex comes from a parallel initialisation (k_queue_init), which replaces
// the clearing of the words.
//
// Word of a vertex outside the tree, b = bits of a neighbour index (kc_host_plan.h):
//   low half   the last arrow taken, the next arrow, those after it (b bits each),
//              then a single 1 that marks the end of the queue
//   high half  departures so far (bit 31 clear)
// In-tree words are the common ones (parent, depth, bit 63).  A departure count
// near its limit sets kErrCountField and the host repeats the wave with the
// walkers of k1_wilson.cu.
#include <algorithm>

#include "kc_common.cuh"
#include "kc_host_plan.h"

namespace kc {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Neighbours of a vertex.  kDeg4 (every degree at most 4): the 16-byte record, so
// that a departure loads one piece of it.
template <bool kDeg4>
struct Nbrs {
    VRec r;
    __device__ __forceinline__ void load(const GraphView &g, int32_t v) { r = load_rec(g.rec + v); }
    __device__ __forceinline__ int32_t pick(uint32_t k, const GraphView &g) const {
        return nbr_of(r, k, g.col);
    }
    __device__ __forceinline__ uint32_t degree() const { return (uint32_t)r.deg; }
};
template <>
struct Nbrs<true> {
    int4 r;
    __device__ __forceinline__ void load(const GraphView &g, int32_t v) { r = __ldg(g.rec4 + v); }
    __device__ __forceinline__ int32_t pick(uint32_t k, const GraphView &) const {
        const int32_t lo = (k & 1u) ? r.y : r.x, hi = (k & 1u) ? r.w : r.z;
        return (k & 2u) ? hi : lo;
    }
    __device__ __forceinline__ uint32_t degree() const {  // -1 past the last neighbour
        return 1u + (r.y >= 0) + (r.z >= 0) + (r.w >= 0);
    }
};

// Words of every tree of the wave: the first `slots` arrows of each vertex, the
// root (if any) in the tree.  A thread keeps one vertex's degree for kInitTrees
// trees.
constexpr int kInitTrees = 8;
__global__ void __launch_bounds__(256) k_queue_init(GraphView g, WaveView w, PhiloxKeys keys,
                                                    uint64_t seed,
                                                    const int64_t *__restrict__ sids,
                                                    int32_t root, int b, int slots) {
    const int64_t n = g.n;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const uint32_t deg = (uint32_t)g.deg[v];
    for (int64_t t0 = (int64_t)blockIdx.y * kInitTrees; t0 < w.B;
         t0 += (int64_t)gridDim.y * kInitTrees) {
        const int64_t t1 = t0 + kInitTrees < w.B ? t0 + kInitTrees : w.B;
        for (int64_t t = t0; t < t1; ++t) {
            uint64_t x;
            if (v == root) {
                x = w_make(-1, 0, true);
                w.ord[t * n] = root;
            } else {
                const uint32_t sample = (uint32_t)sids[t];
                uint32_t q = 1u << (b * (slots + 1));
                for (int j = 0; j < slots; ++j)
                    q |= bounded_draw_k(keys, seed, (uint32_t)v, (uint32_t)j, sample, kTagWalk,
                                        deg)
                         << (b * (j + 1));
                x = q;
            }
            w.word[t * n + v] = x;
        }
    }
}

// Results of a finished (or failed) tree, written by one lane.  A failed tree
// flags -1 like a rejected one, so that no traversal reads its unfinished words.
enum : int { kEndOk = 0, kEndSteps = 1, kEndField = 2 };
template <bool kReject>
__device__ __forceinline__ void finish_tree(const WaveView &w, int64_t t, int end, int64_t steps,
                                            int32_t maxd, volatile int32_t *done_flag) {
    const bool drop = end != kEndOk;
    if (end == kEndField) atomicOr(w.err, kErrCountField);
    if (!kReject && end == kEndSteps) atomicOr(w.err, kErrStepLimit);
    w.steps[t] = drop ? -1 : steps;
    if (!drop) atomicMax(w.maxdepth, maxd);
    if (done_flag) {  // publish the tree: its depth + 1
        __threadfence_system();
        done_flag[t] = drop ? -1 : maxd + 1;
    }
}

// Commits the loop-erased path s .. h (h in the tree at depth dh) along the last
// arrows: depths, parents and the parent-first order from slot pos on.  A group
// of kGroup lanes (mask gm) follows the path; lane j of a chunk of kGroup keeps
// vertex j, full chunks wait at the free end of ord.  Returns its length, -1 when
// it is longer than the vertices left (corrupt state).
template <int kGroup, bool kDeg4>
__device__ __forceinline__ int32_t commit_path(unsigned gm, uint64_t *word, int32_t *ord,
                                               const GraphView &g, int32_t n, uint32_t kmask,
                                               int32_t s, int32_t h, int32_t dh, int32_t pos) {
    constexpr int32_t kIn = kGroup - 1;
    const int lane = threadIdx.x & kIn;
    int32_t len = 0, mine = 0, par = 0, x = s;
    Nbrs<kDeg4> r;
    while (x != h) {
        const uint32_t lo = (uint32_t)word[x];
        r.load(g, x);
        const int32_t px = r.pick(lo & kmask, g);
        if (lane == (len & kIn)) {
            mine = x;
            par = px;
        }
        ++len;
        if ((len & kIn) == 0) {
            if (len > n - pos) return -1;
            ord[n - len + kIn - lane] = mine;
        }
        x = px;
    }
    if (len > n - pos) return -1;
    // nearest the tree first: vertex j gets depth dh + len - j and slot
    // pos + len - 1 - j
    int32_t j = (len & ~kIn) + lane;
    __syncwarp(gm);
    if (j < len) {
        word[mine] = w_make(par, (uint32_t)(dh + len - j), true);
        ord[pos + len - 1 - j] = mine;
    }
    for (j -= kGroup; j >= lane; j -= kGroup) {
        __syncwarp(gm);
        const int32_t y = ord[n - 1 - j];
        r.load(g, y);
        const int32_t py = r.pick((uint32_t)word[y] & kmask, g);
        __syncwarp(gm);
        word[y] = w_make(py, (uint32_t)(dh + len - j), true);
        ord[pos + len - 1 - j] = y;
    }
    __syncwarp(gm);
    return len;
}

// One tree per group of kGroup lanes, 32 / kGroup trees per warp.  The lanes of a
// group follow their walk together (one address, one transaction) and share the
// work around it: starts are looked up and paths committed kGroup vertices at a
// time, and a refill draws an arrow per lane.  All walks of a warp depart in
// lockstep until one of them meets the tree; when one queue is empty, every
// walk's vertex is refilled, which costs the warp the same.
//
// Measured (GB300, perturbed grids, ncu): 32 warp instructions and 187 cycles a
// departure with one tree per warp on an otherwise idle SM, of which 40 wait for
// memory (L1 serves 95%); the 32 lockstep walkers of one tree (k_wilson_warp) take
// about 650 cycles, a walker per lane (k_wilson) about 1100.  Walk of 500 trees of a
// 40000-vertex grid: 299 (k_wilson_warp) -> 126 ms; of 4522 trees of the 350x350 grid
// under a cap of 13 n departures: 1640 (k_wilson) -> 350 ms.  The word that held the
// next target itself, with the queue behind it, made the load chain shorter and the
// kernel slower: 52 instructions, 250 cycles.
template <int kGroup, bool kDeg4, bool kReject>
__device__ __forceinline__ void walk_trees(const GraphView &g, const WaveView &w,
                                           const PhiloxKeys &keys, uint64_t seed, uint32_t sample,
                                           int64_t t, bool on, int bits, int slots,
                                           int64_t step_cap, volatile int32_t *done_flag) {
    constexpr bool kOne = kGroup == 32;
    constexpr unsigned kIn = kGroup - 1;
    const unsigned lane = threadIdx.x & kIn;
    const unsigned gshift = threadIdx.x & ~kIn;
    const unsigned gm = kOne ? kFull : ((1u << (kGroup & 31)) - 1u) << gshift;
    const int32_t n = (int32_t)g.n;
    const int b = kDeg4 ? 2 : bits;
    const uint32_t kmask = (1u << b) - 1u;
    const uint32_t last = 2u << (2 * b);  // a queue below this holds one more arrow
    // what follows is the same in every lane of a group; on: its tree is being walked
    const int64_t tt = on ? t : 0;
    uint64_t *word = w.word + tt * g.n;
    int32_t *ord = w.ord + tt * g.n;
    int64_t steps = 0;  // departures before the last refill or path
    uint32_t more = 0;  // and since
    int32_t pos = w.pos0, maxd = 0;
    int32_t s = 0, base = -kGroup;  // start of the walk; chunk of starts looked up
    unsigned todo = 0;              // its vertices that were outside the tree
    int32_t u = 0;                  // the walk's vertex, its word and neighbours
    uint32_t lo = 0, hi = 0;
    Nbrs<kDeg4> ra{}, rb{};
    int end = kEndOk;
    bool start = on, hit = false;

    // One departure of every walk, from the vertex of neighbours rc to that of rn;
    // whether some walk has to leave the lockstep.
    auto depart = [&](const Nbrs<kDeg4> &rc, Nbrs<kDeg4> &rn) -> bool {
        int32_t v = 0;
        uint64_t x = 0;
        if (kOne || on) {
            v = rc.pick((lo >> b) & kmask, g);
            x = word[v];
            rn.load(g, v);
        }
        const bool empty = (kOne || on) && lo < last;
        lo >>= b;
        ++hi;
        if (kOne ? empty : __any_sync(kFull, empty)) {
            // lane j draws the arrow after the next j
            uint32_t d = 0;
            if (lane < (unsigned)slots)
                d = bounded_draw_k(keys, seed, (uint32_t)u, hi + lane, sample, kTagWalk,
                                   rc.degree())
                    << (b * (lane + 1));
            if (kOne) {
                d = __reduce_or_sync(kFull, d);
            } else {
#pragma unroll
                for (int o = kGroup / 2; o > 0; o >>= 1) d |= __shfl_xor_sync(kFull, d, o);
            }
            lo = (lo & kmask) | d | (1u << (b * (slots + 1)));
            steps += more + 1;
            more = (uint32_t)-1;
            if (hi + slots >= kWalkCountMask) end = kEndField;
            if (steps > step_cap) end = kEndSteps;
            if (!on) end = kEndOk;
        } else if (kOne) {
            __syncwarp();  // every lane has read the words of the last departure
        }
        if (kOne || on) {
            word[u] = (uint64_t)lo | ((uint64_t)hi << 32);
            ++more;
            u = v;
            lo = (uint32_t)x;
            hi = (uint32_t)(x >> 32);
            hit = (int32_t)hi < 0;
        }
        const bool leave = hit || end != kEndOk;
        return kOne ? leave : __any_sync(kFull, leave);
    };

    for (;;) {
        // ---- the next start outside the tree, kGroup vertices at a time
        if (start) {
            start = false;
            for (;;) {
                while (!todo && base + kGroup < n) {
                    base += kGroup;
                    bool out = false;
                    if (base + (int32_t)lane < n) out = !w_in_tree(word[base + lane]);
                    todo = (__ballot_sync(gm, out) & gm) >> gshift;
                }
                if (!todo) {
                    on = false;
                    if (steps > step_cap) end = kEndSteps;
                    if (lane == 0) finish_tree<kReject>(w, t, end, steps, maxd, done_flag);
                    end = kEndOk;
                    break;
                }
                s = base + __ffs(todo) - 1;
                todo &= todo - 1;
                const uint64_t x = word[s];
                if (w_in_tree(x)) continue;  // an earlier path of this chunk took it
                u = s;
                lo = (uint32_t)x;
                hi = (uint32_t)(x >> 32);
                ra.load(g, s);
                break;
            }
        }
        if (kOne ? !on : !__any_sync(kFull, on)) break;
        // ---- departures
        for (;;) {
            if (depart(ra, rb)) {
                ra = rb;
                break;
            }
            if (depart(rb, ra)) break;
        }
        // ---- walks that met the tree or were given up
        __syncwarp();
        if (on && (hit || end != kEndOk)) {
            int32_t len = 0;
            if (end == kEndOk) {
                steps += more;
                more = 0;
                hit = false;
                start = true;
                hi &= 0x7FFFFFFFu;
                len = commit_path<kGroup, kDeg4>(gm, word, ord, g, n, kmask, s, u, (int32_t)hi,
                                                 pos);
                if (len < 0) end = kEndField;
            }
            if (end != kEndOk) {
                if (lane == 0) finish_tree<kReject>(w, t, end, 0, 0, done_flag);
                end = kEndOk;
                on = hit = start = false;
            } else {
                pos += len;
                maxd = max(maxd, (int32_t)hi + len);
            }
        }
        __syncwarp();
    }
}

template <int kGroup, bool kDeg4, bool kReject>
__global__ void __launch_bounds__(32, kGroup == 32 ? 32 : 24)
    k_wilson_queue(GraphView g, WaveView w, PhiloxKeys keys, uint64_t seed,
                   const int64_t *__restrict__ sids, int bits, int slots, int64_t step_cap,
                   volatile int32_t *done_flag) {
    const int64_t t = (int64_t)blockIdx.x * (32 / kGroup) + threadIdx.x / kGroup;
    const bool on = t < w.B;
    walk_trees<kGroup, kDeg4, kReject>(g, w, keys, seed, (uint32_t)sids[on ? t : 0], t, on, bits,
                                       slots, step_cap, done_flag);
}

// block j takes tree mw.entry[j].y of graph mw.entry[j].x
__global__ void __launch_bounds__(32, 32) k_wilson_queue_multi(MultiWalk mw) {
    const int e = mw.entry[blockIdx.x].x;
    const int64_t t = mw.entry[blockIdx.x].y;
    const GraphView g = mw.graphs[e];
    const WaveView w = mw.waves[e];
    const uint64_t seed = mw.seeds[e];
    const PhiloxKeys keys = philox_keys(seed);
    const uint32_t sample = (uint32_t)mw.sids[e][t];
    const int bits = mw.queue_bits[e];
    const int slots = kc_host::queue_slots(bits);
    if (g.rec4)
        walk_trees<32, true, false>(g, w, keys, seed, sample, t, true, bits, slots,
                                    mw.step_caps[e], nullptr);
    else
        walk_trees<32, false, false>(g, w, keys, seed, sample, t, true, bits, slots,
                                     mw.step_caps[e], nullptr);
}

}  // namespace

cudaError_t launch_queue_init(const GraphView &g, WaveView w, uint64_t seed, const int64_t *sids,
                              int32_t root, int bits, int first_slots, cudaStream_t s) {
    const dim3 grid((unsigned)((g.n + 255) / 256),
                    (unsigned)std::min<int64_t>((w.B + kInitTrees - 1) / kInitTrees, 65535));
    k_queue_init<<<grid, 256, 0, s>>>(g, w, host_keys(seed), seed, sids, root, bits,
                                      std::min(first_slots, kc_host::queue_slots(bits)));
    return cudaGetLastError();
}

namespace {
template <int kGroup, bool kDeg4>
void launch_group(const GraphView &g, const WaveView &w, uint64_t seed, const int64_t *sids,
                  int bits, int64_t step_cap, bool reject, cudaStream_t s, int32_t *done_flag) {
    const PhiloxKeys K = host_keys(seed);
    const int slots = std::min(kc_host::queue_slots(bits), kGroup);
    const unsigned blocks = (unsigned)((w.B * kGroup + 31) / 32);
    if (reject)
        k_wilson_queue<kGroup, kDeg4, true><<<blocks, 32, 0, s>>>(g, w, K, seed, sids, bits, slots,
                                                                  step_cap, done_flag);
    else
        k_wilson_queue<kGroup, kDeg4, false><<<blocks, 32, 0, s>>>(g, w, K, seed, sids, bits,
                                                                   slots, step_cap, done_flag);
}
}  // namespace

cudaError_t launch_wilson_queue(const GraphView &g, WaveView w, uint64_t seed,
                                const int64_t *sids, int bits, int64_t step_cap, bool reject,
                                int64_t num_sms, cudaStream_t s, int32_t *done_flag) {
    const int group = kc_host::queue_group(w.B, num_sms);
    const bool deg4 = g.rec4 != nullptr;
    auto *launch = group == 32 ? (deg4 ? launch_group<32, true> : launch_group<32, false>)
                               : (deg4 ? launch_group<16, true> : launch_group<16, false>);
    launch(g, w, seed, sids, bits, step_cap, reject, s, done_flag);
    return cudaGetLastError();
}

cudaError_t launch_wilson_queue_multi(const MultiWalk &mw, cudaStream_t s) {
    if (mw.count <= 0) return cudaSuccess;
    k_wilson_queue_multi<<<(unsigned)mw.count, 32, 0, s>>>(mw);
    return cudaGetLastError();
}

}  // namespace kc
