// Wilson's loop-erased-walk sampler (Sec. 2.2), one walker per tree with the
// arrows drawn ahead.  The trees, step counts and parent-first orders are those
// of k1_wilson.cu: vertex u's k-th arrow is bounded(seed, u, k, sample, WALK,
// deg u), and by cycle popping neither the start order nor the walker matters.
//
// What bounds a sequential walker is the chain of one departure: load the word
// of the vertex, ten dependent Philox rounds, select the neighbour, load its
// word.  Here the word of a vertex outside the tree holds the target of its next
// departure and a queue of the arrows after it as neighbour indices, so the walk
// is a pointer chase: the next word is requested at once, and behind the walker
// the vertex left gets its new target (a bit field and a select) while that load
// is in flight.  An empty queue is refilled by the warp, one arrow per lane.  The
// first queue of every vertex comes from a parallel initialisation
// (k_queue_init), which replaces the clearing of the words.
//
// Word of a vertex outside the tree, b = bits of a neighbour index (kc_host_plan.h):
//   low half   target of the next departure
//   high half  bits [0, 17): the last arrow taken, the next arrow, those after it
//              (b bits each), then a single 1 that marks the end of the queue;
//              bits [17, 31): departures so far; bit 31 clear
// In-tree words are the common ones (parent, depth, bit 63).  A departure count
// that its field may not hold sets kErrCountField and the host repeats the wave
// with the walkers of k1_wilson.cu.
#include <algorithm>

#include "kc_common.cuh"
#include "kc_host_plan.h"

namespace kc {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr uint32_t kQueue = (1u << kc_host::kQueueWidth) - 1u;
constexpr uint32_t kOneMore = 1u << kc_host::kQueueWidth;  // one departure in the high half
constexpr uint32_t kMostDepartures = (1u << (31 - kc_host::kQueueWidth)) - 1u;

// Words of every tree of the wave: the first `slots` arrows of each vertex, the
// root (if any) in the tree.  A thread keeps one vertex's record for kInitTrees
// trees.
constexpr int kInitTrees = 8;
__global__ void __launch_bounds__(256) k_queue_init(GraphView g, WaveView w, PhiloxKeys keys,
                                                    uint64_t seed,
                                                    const int64_t *__restrict__ sids,
                                                    int32_t root, int b, int slots) {
    const int64_t n = g.n;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const VRec r = load_rec(g.rec + v);
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
                uint32_t q = 1u << (b * (slots + 1)), first = 0;
                for (int j = 0; j < slots; ++j) {
                    const uint32_t d = bounded_draw_k(keys, seed, (uint32_t)v, (uint32_t)j,
                                                      sample, kTagWalk, (uint32_t)r.deg);
                    q |= d << (b * (j + 1));
                    first = j == 0 ? d : first;
                }
                x = (uint64_t)(uint32_t)nbr_of<false>(r, first, g.col) | ((uint64_t)q << 32);
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
                                               const VRec *__restrict__ rec,
                                               const int32_t *__restrict__ col, int32_t n,
                                               uint32_t kmask, int32_t s, int32_t h, int32_t dh,
                                               int32_t pos) {
    constexpr int32_t kIn = kGroup - 1;
    const int lane = threadIdx.x & kIn;
    int32_t len = 0, mine = 0, par = 0, x = s;
    while (x != h) {
        const uint32_t hi = (uint32_t)(word[x] >> 32);
        const VRec r = load_rec(rec + x);
        const int32_t px = nbr_of<kDeg4>(r, hi & kmask, col);
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
        const int32_t py =
            nbr_of<kDeg4>(load_rec(rec + y), (uint32_t)(word[y] >> 32) & kmask, col);
        __syncwarp(gm);
        word[y] = w_make(py, (uint32_t)(dh + len - j), true);
        ord[pos + len - 1 - j] = y;
    }
    __syncwarp(gm);
    return len;
}

// One tree per group of kGroup lanes, 32 / kGroup trees per warp.
//
// Measured (GB300, perturbed grids, ncu): about 52 warp instructions and 250
// cycles a departure with one tree per warp on an otherwise idle SM, of which 60
// wait for L1; 32 concurrent walkers of one tree (k_wilson_warp) take about 650.
// 1000 trees of the 350x350 grid: 1330 -> 661 ms; 4522 trees of it under a cap of
// 13 n departures: 1640 (k_wilson, one tree per lane) -> 508 ms.  With 28 trees
// an SM the schedulers issue in 0.7 of their slots, so the rest is instructions.
//  The lanes of a
// group follow their walk together (one address, one transaction) and share the
// work around it: starts are looked up and paths committed kGroup vertices at a
// time, and a refill draws an arrow per lane.  All walks of a warp depart in
// lockstep until one of them meets the tree; when one queue is empty, every
// walk's vertex is refilled, which costs the warp the same.
// kMulti (with kGroup 32): block j takes tree mw.entry[j].y of graph
// mw.entry[j].x.
struct QueueShape {
    int b, slots;
};
template <int kGroup, bool kDeg4, bool kMulti, bool kReject>
__global__ void __launch_bounds__(32, kGroup == 32 ? 28 : (kGroup == 16 ? 20 : 24)) k_wilson_queue(
    GraphView g_in, WaveView w_in, PhiloxKeys keys_in, uint64_t seed_in,
    const int64_t *__restrict__ sids_in, QueueShape shape_in, int64_t step_cap_in,
    volatile int32_t *done_flag, MultiWalk mw) {
    constexpr int kTrees = 32 / kGroup;
    constexpr unsigned kIn = kGroup - 1;
    const unsigned lane = threadIdx.x & kIn;
    const unsigned gshift = threadIdx.x & ~kIn;
    const unsigned gm = kGroup == 32 ? kFull : ((1u << (kGroup & 31)) - 1u) << gshift;
    const int e = kMulti ? mw.entry[blockIdx.x].x : 0;
    const int64_t t = kMulti ? (int64_t)mw.entry[blockIdx.x].y
                             : (int64_t)blockIdx.x * kTrees + gshift / kGroup;
    const uint64_t seed = kMulti ? mw.seeds[e] : seed_in;
    const PhiloxKeys keys = kMulti ? philox_keys(seed) : keys_in;
    const int64_t step_cap = kMulti ? mw.step_caps[e] : step_cap_in;
    const int64_t n64 = kMulti ? mw.graphs[e].n : g_in.n;
    const VRec *__restrict__ rec = kMulti ? mw.graphs[e].rec : g_in.rec;
    const int32_t *__restrict__ col = kMulti ? mw.graphs[e].col : g_in.col;
    const WaveView w = kMulti ? mw.waves[e] : w_in;
    const int b = kMulti ? mw.queue_bits[e] : shape_in.b;
    const int slots = kMulti ? kc_host::queue_slots(b) : shape_in.slots;
    const int32_t n = (int32_t)n64;
    const uint32_t kmask = (1u << b) - 1u;
    // what follows is the same in every lane of a group
    bool on = kTrees == 1 || t < w.B;  // the tree is still being walked
    const int64_t tt = on ? t : 0;
    uint64_t *word = w.word + tt * n64;
    int32_t *ord = w.ord + tt * n64;
    const uint32_t sample = (uint32_t)(kMulti ? mw.sids[e][tt] : sids_in[tt]);
    int64_t steps = 0;           // departures before the last refill or path
    uint32_t more = 0;           // and since
    int32_t pos = w.pos0, maxd = 0;
    int32_t s = 0, base = -kGroup;  // start of the walk; chunk of starts looked up
    unsigned todo = 0;              // its vertices that were outside the tree
    int32_t u = 0, lo = 0;          // the walk's vertex, its word and record
    uint32_t hi = 0;
    VRec ra, rb;
    ra.deg = rb.deg = 1;
    int end = kEndOk;
    bool start = on, hit = false;

    // One departure of every walk, from the vertex of record rc to that of rn;
    // whether some walk has to leave the lockstep.
    auto depart = [&](const VRec &rc, VRec &rn) -> bool {
        int32_t v = 0;
        uint64_t x = 0;
        uint32_t left = 0, next = 0, count = 0;
        if (kTrees == 1 || on) {
            v = lo;
            x = word[v];
            rn = load_rec(rec + v);
            const uint32_t queue = hi & kQueue;
            left = queue >> b;  // the arrow taken, then the rest
            next = left >> b;
            count = (hi ^ queue) + kOneMore;
        }
        uint32_t k = next & kmask;
        const bool empty = (kTrees == 1 || on) && next == 1u;  // only the end mark
        if (kTrees == 1 ? empty : __any_sync(kFull, empty)) {
            // lane j draws the arrow after the next j
            const uint32_t c = count >> kc_host::kQueueWidth;
            uint32_t d = 0;
            if (lane < (unsigned)slots)
                d = bounded_draw_k(keys, seed, (uint32_t)u, c + lane, sample, kTagWalk,
                                   (uint32_t)rc.deg)
                    << (b * (lane + 1));
            if (kGroup == 32) {
                d = __reduce_or_sync(kFull, d);
            } else {
#pragma unroll
                for (int o = kGroup / 2; o > 0; o >>= 1) d |= __shfl_xor_sync(kFull, d, o);
            }
            left = (left & kmask) | d | (1u << (b * (slots + 1)));
            k = (d >> b) & kmask;
            steps += more + 1;
            more = (uint32_t)-1;
            if (c + slots > kMostDepartures) end = kEndField;
            if (steps > step_cap) end = kEndSteps;
            if (!on) end = kEndOk;
        } else if (kTrees == 1) {
            __syncwarp();  // every lane has read the words of the last departure
        }
        if (kTrees == 1 || on) {
            const int32_t target = nbr_of<kDeg4>(rc, k, col);
            word[u] = (uint64_t)(uint32_t)target | ((uint64_t)(count + left) << 32);
            ++more;
            u = v;
            lo = w_next(x);
            hi = (uint32_t)(x >> 32);
            hit = (int32_t)hi < 0;
        }
        const bool leave = hit || end != kEndOk;
        return kTrees == 1 ? leave : __any_sync(kFull, leave);
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
                lo = w_next(x);
                hi = (uint32_t)(x >> 32);
                ra = load_rec(rec + s);
                break;
            }
        }
        if (kTrees == 1 ? !on : !__any_sync(kFull, on)) break;
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
                len = commit_path<kGroup, kDeg4>(gm, word, ord, rec, col, n, kmask, s, u,
                                                 (int32_t)hi, pos);
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
    const QueueShape q{bits, std::min(kc_host::queue_slots(bits), kGroup)};
    const unsigned blocks = (unsigned)((w.B * kGroup + 31) / 32);
    if (reject)
        k_wilson_queue<kGroup, kDeg4, false, true><<<blocks, 32, 0, s>>>(
            g, w, K, seed, sids, q, step_cap, done_flag, MultiWalk{});
    else
        k_wilson_queue<kGroup, kDeg4, false, false><<<blocks, 32, 0, s>>>(
            g, w, K, seed, sids, q, step_cap, done_flag, MultiWalk{});
}
}  // namespace

cudaError_t launch_wilson_queue(const GraphView &g, WaveView w, uint64_t seed,
                                const int64_t *sids, int bits, int64_t step_cap, bool reject,
                                int64_t num_sms, cudaStream_t s, int32_t *done_flag) {
    const int group = kc_host::queue_group(w.B, num_sms);
    const bool deg4 = bits <= 2;
    auto *launch = group == 32 ? (deg4 ? launch_group<32, true> : launch_group<32, false>)
                 : group == 16 ? (deg4 ? launch_group<16, true> : launch_group<16, false>)
                               : (deg4 ? launch_group<8, true> : launch_group<8, false>);
    launch(g, w, seed, sids, bits, step_cap, reject, s, done_flag);
    return cudaGetLastError();
}

cudaError_t launch_wilson_queue_multi(const MultiWalk &mw, cudaStream_t s) {
    if (mw.count <= 0) return cudaSuccess;
    k_wilson_queue<32, false, true, false><<<(unsigned)mw.count, 32, 0, s>>>(
        GraphView{}, WaveView{}, PhiloxKeys{}, 0, nullptr, QueueShape{1, 1}, 0, nullptr, mw);
    return cudaGetLastError();
}

}  // namespace kc
