// Spanning trees of low-diameter graphs by cycle popping, and f(tau) of each tree
// in the same block (Sec. 2.2; Theorem 3).
//
// Wilson's algorithm pops the cycles of stacks of arrows (vertex u's k-th arrow is
// bounded(seed, u, k, sample, WALK, deg u)); popping them in any order gives the
// same tree and the same number of arrows.  Here a block takes a tree: every
// vertex shows its first arrow, all cycles of that map are found and their
// vertices shown their next arrows, and so on until none is left.  On a
// low-diameter graph the first map holds most of the tree -- a random graph of
// 2000 vertices pops about 0.5 n arrows in some 20 rounds, a power-law graph of a
// million 0.09 n in 10 to 80 -- where a walk is a chain of n loads and more.
//
// A cycle is found by its leader, the smallest active vertex on it (active: its
// arrow is new; every cycle holds one).  An active vertex a follows the arrows
// until a settled vertex (one known to lead to the root: then so does a, and
// its path is settled), an active vertex below a (which then leads, if anything
// does), a itself, or an active vertex met before (Brent's rule: a cycle of larger
// vertices that does not hold a).  Settled paths are never followed again, so all
// rounds together settle each vertex once.
//
// Once few vertices are active, the round works on the map that they form: each
// follows the arrows to the next active vertex only, and that map is squared until
// its images are the vertices on its cycles (contracted_round); each of those lists
// its own piece of the cycle.  A round of some 50 active vertices then costs its
// longest piece where the leaders' loops went around several times: 2000 trees of a
// random graph of 2000 vertices (kc_wilson_noalloc) 2.62 -> 2.23 ms, 1.4 by now.
//
// k_pop_small keeps the tree in shared memory: 14 bytes a vertex.  Larger trees
// stay in memory: the first arrows (k_first_arrows) and the cycles of the first map
// (k_first_cycles) are passes over all vertices of all trees, the rounds after it,
// which touch a tenth of the vertices where the root is a hub, a block per tree
// (k_pop_rounds); the traversal is that of k2_parents.cu.  What bounds it is the
// rate of random sectors, about ten a vertex with the traversal.
//
// Measured (GB300, power-law graphs of mean degree 17, against 32 walkers a tree
// and their traversal): 2 million vertices, 384 trees 830 -> 140 ms (rounds 43,
// first cycles 16, first arrows 5; traversal 65, tau0 scan 10); 10000 vertices in
// shared memory, 500 trees 5.3 -> 0.9 ms.  Random graph of 2000 vertices, 2000 trees:
// 3.8 -> 1.4 ms.
#include <algorithm>
#include <atomic>

#include "kc_common.cuh"
#include "kc_host_plan.h"

namespace kc {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Vertex word in shared memory: target (16 bits), pops (13), on a cycle, settled,
// active
constexpr uint32_t kActive = 1u << 31;
constexpr uint32_t kSettled = 1u << 30;
constexpr uint32_t kOnCycle = 1u << 29;
constexpr uint32_t kTarget = 0xFFFFu;
constexpr uint32_t kSmallMostPops = 0x1FFFu;

// Squares the map `next` of the `active` vertices list[] (-1: leads to the root)
// until every image lies on a cycle of it.  The whole block calls; each thread holds
// up to kHold vertices.
constexpr int kHold = 4;
template <int kThreads, class Vertex, class Hop>
__device__ __forceinline__ void square_map(const Vertex *list, uint32_t active, Hop *next) {
    const Hop none = (Hop)-1;
    volatile Hop *map = next;
    const int rounds = 32 - __clz(active);  // 2^rounds > active
    const bool warp = active <= 32 * kHold;  // one warp holds them all
    const uint32_t step = warp ? 32 : kThreads;
    if (!warp || threadIdx.x < 32) {
        Vertex a[kHold];
        Hop h[kHold];
#pragma unroll
        for (int j = 0; j < kHold; ++j) {
            const uint32_t i = threadIdx.x + j * step;
            a[j] = 0;
            h[j] = none;
            if (i < active) {
                a[j] = list[i];
                h[j] = map[a[j]];
            }
        }
        for (int r = 0; r < rounds; ++r) {
#pragma unroll
            for (int j = 0; j < kHold; ++j) {
                if (j * step >= active) break;
                if (h[j] != none) h[j] = map[h[j]];
            }
            if (warp) __syncwarp(); else __syncthreads();
#pragma unroll
            for (int j = 0; j < kHold; ++j) {
                if (j * step >= active) break;
                if (threadIdx.x + j * step < active) map[a[j]] = h[j];
            }
            if (warp) __syncwarp(); else __syncthreads();
        }
    }
    __syncthreads();
}

// The length of the cycle that active vertex a leads, or 0 (see above).
__device__ __forceinline__ uint32_t led_cycle(volatile uint32_t *nx, uint32_t a) {
    uint32_t x = nx[a] & kTarget;
    uint32_t saved = 0xFFFFFFFFu, met = 0, power = 1, len = 1;
    for (;; ++len) {
        const uint32_t w = nx[x];
        if (w >= kSettled) {
            if (w & kSettled) break;
            if (x <= a) return x == a ? len : 0;
            if (x == saved) return 0;
            if (++met == power) {
                saved = x;
                power <<= 1;
                met = 0;
            }
        }
        x = w & kTarget;
    }
    // a leads to the root: settle its path (others may settle parts of it too)
    x = a;
    for (uint32_t w = nx[x]; !(w & kSettled); w = nx[x]) {
        nx[x] = w | kSettled;
        x = w & kTarget;
    }
    return 0;
}

// kKind: kFused evaluates f; kTrees leaves the parents in task.par only (whose row
// holds the two lists meanwhile) and needs 6 bytes a vertex (4, past
// kPopContractMax, without contracted rounds); kTreesCsr does so
// from the CSR arrays alone, and marks a tree that it cannot finish kPopRedo
// instead of raising an error.
enum : int { kFused = 0, kTrees = 1, kTreesCsr = 2 };
template <int kThreads, bool kMulti, int kKind>
__global__ void __launch_bounds__(kThreads,
                                  kThreads <= 128 ? 10 : (kThreads <= 256 ? 5 : 1024 / kThreads))
    k_pop_small(PopTask one, const PopTask *__restrict__ tasks, const int2 *__restrict__ entry) {
    const int64_t t = kMulti ? (int64_t)entry[blockIdx.x].y : (int64_t)blockIdx.x;
    const PopTask task = kMulti ? tasks[entry[blockIdx.x].x] : one;
    const GraphView &g = task.g;
    const uint32_t n = (uint32_t)g.n, root = (uint32_t)task.root;
    const uint32_t sample = (uint32_t)(kKind == kTreesCsr ? task.first_sid + t : task.sids[t]);
    const uint32_t tid = threadIdx.x;
    const VRec *__restrict__ rec = g.rec;

    extern __shared__ uint32_t smem[];
    uint32_t *nx = smem;       // [n] the map
    uint32_t *acc = smem + n;  // [n] the two lists of active vertices; then reports, jumps
    uint32_t *vol = smem + 2 * n;
    uint16_t *size = reinterpret_cast<uint16_t *>(smem + 3 * n);
    uint16_t *list = kKind == kFused ? reinterpret_cast<uint16_t *>(acc)
                                     : reinterpret_cast<uint16_t *>(task.par + t * n);
    uint16_t *fresh = list + n;
    uint16_t *next = reinterpret_cast<uint16_t *>(kKind == kFused ? vol : smem + n);  // [n]
    const bool contract = kKind == kFused || n <= kc_host::kPopContractMax;
    __shared__ uint32_t s_count[2];
    __shared__ unsigned long long s_f;

    // arrow number `count` of v
    auto arrow = [&](uint32_t v, uint32_t count) {
        if (kKind == kTreesCsr) {
            const int64_t off = g.row_off[v];
            const uint32_t k = bounded_draw_k(task.keys, task.seed, v, count, sample, kTagWalk,
                                              (uint32_t)(g.row_off[v + 1] - off));
            return (uint32_t)g.col[off + k];
        }
        const VRec r = load_rec(rec + v);
        const uint32_t k = bounded_draw_k(task.keys, task.seed, v, count, sample, kTagWalk,
                                          (uint32_t)r.deg);
        return (uint32_t)nbr_of(r, k, g.col);
    };
    for (uint32_t v = tid; v < n; v += kThreads) {
        uint32_t x = root | kSettled;
        if (v != root && (int32_t)v != task.fixed) x = arrow(v, 0) | kActive;
        nx[v] = x;
    }
    if (tid < 2) s_count[tid] = 0;
    if (tid == 0) s_f = 0;
    __syncthreads();

    // ---- rounds: leaders list their cycles, the cycles' arrows are replaced
    uint32_t active = n;  // round 0: every vertex
    int64_t pops = 0;
    int end = 0;
    for (int round = 0;; ++round) {
        if (round > 0 && contract && active <= kHold * kThreads) {
            volatile uint32_t *vx = nx;
            uint32_t len[kHold];
            for (int j = 0; j < kHold; ++j) {
                const uint32_t i = tid + j * kThreads;
                if (i >= active) break;
                const uint32_t a = list[i];
                // three hops a test: every word's target is a vertex, so a hop
                // past the end is only wasted, and a test between two hops would
                // wait for the first
                uint32_t x = vx[a] & kTarget, w, l = 1;
                for (;; l += 3) {
                    w = vx[x];
                    const uint32_t x1 = w & kTarget, w1 = vx[x1];
                    const uint32_t x2 = w1 & kTarget, w2 = vx[x2];
                    if ((w | w1 | w2) < kSettled) {
                        x = w2 & kTarget;
                        continue;
                    }
                    if (w >= kSettled) break;
                    const bool first = w1 >= kSettled;
                    x = first ? x1 : x2;
                    w = first ? w1 : w2;
                    l += first ? 1 : 2;
                    break;
                }
                len[j] = l;
                next[a] = (w & kSettled) ? (uint16_t)0xFFFFu : (uint16_t)x;
            }
            __syncthreads();
            square_map<kThreads>(list, active, next);
            for (uint32_t i = tid; i < active; i += kThreads) {
                const uint32_t h = next[list[i]];
                if (h != 0xFFFFu) vx[h] = vx[h] | kOnCycle;
            }
            __syncthreads();
            for (int j = 0; j < kHold; ++j) {
                const uint32_t i = tid + j * kThreads;
                if (i >= active) break;
                uint32_t x = list[i];
                if (vx[x] & kOnCycle) {  // its piece of the cycle
                    const uint32_t at = atomicAdd(&s_count[round & 1], len[j]);
                    for (uint32_t k = 0; k < len[j]; ++k) {
                        fresh[at + k] = (uint16_t)x;
                        x = vx[x] & kTarget;
                    }
                } else if (next[x] == 0xFFFFu) {  // its piece of a path to the root
                    for (uint32_t k = 0; k < len[j]; ++k) {
                        const uint32_t w = vx[x];
                        vx[x] = w | kSettled;
                        x = w & kTarget;
                    }
                }
            }
        } else {
            for (uint32_t i = tid; i < active; i += kThreads) {
                const uint32_t a = round == 0 ? i : list[i];
                if (nx[a] & kSettled) continue;
                const uint32_t len = led_cycle(nx, a);
                if (len == 0) continue;
                uint32_t x = a, at = atomicAdd(&s_count[round & 1], len);
                do {
                    fresh[at++] = (uint16_t)x;
                    x = nx[x] & kTarget;
                } while (x != a);
            }
        }
        __syncthreads();
        const uint32_t found = s_count[round & 1];
        for (uint32_t i = tid; i < active; i += kThreads) {
            const uint32_t a = round == 0 ? i : list[i];
            nx[a] &= ~(kActive | kOnCycle);
        }
        if (tid == 0) s_count[(round + 1) & 1] = 0;
        pops += found;
        if (pops + (int64_t)n - task.placed > task.step_cap) {  // also of a first map that is a tree
            end = kErrStepLimit;
            break;
        }
        if (found == 0) break;
        __syncthreads();
        bool full = false;
        for (uint32_t i = tid; i < found; i += kThreads) {
            const uint32_t v = fresh[i];
            const uint32_t c = ((nx[v] >> 16) & kSmallMostPops) + 1;
            nx[v] = arrow(v, c) | (c << 16) | kActive;
            full = full || c >= kSmallMostPops;
        }
        if (__syncthreads_or(full)) {
            end = kErrCountField;
            break;
        }
        active = found;
        uint16_t *const swap = list;
        list = fresh;
        fresh = swap;
    }
    __syncthreads();
    if (end) {  // uniform
        if (tid == 0) {
            if (kKind != kTreesCsr) atomicOr(task.err, (uint32_t)end);
            task.steps[t] = kKind == kTreesCsr ? kPopRedo : -1;
        }
        return;
    }
    if (tid == 0) task.steps[t] = pops + (int64_t)n - task.placed;
    if (kKind != kFused || task.par)
        for (uint32_t v = tid; v < n; v += kThreads)
            task.par[t * n + v] = v == root ? -1 : (int32_t)(nx[v] & kTarget);
    if constexpr (kKind == kFused) {
        // ---- sizes, volumes and preorder.  acc of a vertex: unreported children
        // (high half) and sizes reported (low half); the child that reports last goes
        // on with its parent.  After its own report it holds the vertex's preorder
        // relative to an ancestor: offset (high half) and that ancestor (low half).
        for (uint32_t v = tid; v < n; v += kThreads) {
            acc[v] = 0;
            vol[v] = (uint32_t)g.deg[v];
        }
        __syncthreads();
        for (uint32_t v = tid; v < n; v += kThreads)
            if (v != root) atomicAdd(&acc[nx[v] & kTarget], 1u << 16);
        __syncthreads();
        for (uint32_t v = tid; v < n; v += kThreads) {
            if (*(volatile uint32_t *)&acc[v] != 0u) continue;  // has children
            uint32_t x = v, sx = 1;
            while (x != root) {
                const uint32_t p = nx[x] & kTarget;
                size[x] = (uint16_t)sx;
                atomicAdd(&vol[p], *(volatile uint32_t *)&vol[x]);
                __threadfence_block();
                const uint32_t old = atomicAdd(&acc[p], sx - (1u << 16));
                acc[x] = (((old & 0xFFFFu) + 1u) << 16) | p;
                if ((old >> 16) != 1u) break;  // siblings still to report
                __threadfence_block();
                sx = 1u + (old & 0xFFFFu) + sx;
                x = p;
            }
        }
        __syncthreads();
        if (tid == 0) acc[root] = root;
        __syncthreads();
        // pointer jumping in place: a pair is read and written whole, and holds at
        // any time
        for (uint32_t v = tid; v < n; v += kThreads) {
            volatile uint32_t *pairs = acc;
            uint32_t p = pairs[v];
            while ((p & kTarget) != root) {
                const uint32_t q = pairs[p & kTarget];
                p = (((p >> 16) + (q >> 16)) << 16) | (q & kTarget);
                pairs[v] = p;
            }
        }
        __syncthreads();

        // ---- f: every vertex walks up tau0 (as k_ttf_scan)
        long long contrib = 0;
        for (uint32_t v = tid; v < n; v += kThreads) {
            if (v == root) continue;
            const uint32_t inv = acc[v] >> 16;
            long long q = 0;
            uint32_t x = v;
            for (int it = 0; x != root && it <= g.ecc; ++it) {
                const uint32_t p0x = (uint32_t)g.p0[x];
                if ((nx[x] & kTarget) == p0x) {
                    if (inv - (acc[x] >> 16) < size[x]) q += g.twom - (int64_t)vol[x];
                } else if (p0x != root && (nx[p0x] & kTarget) == x) {
                    if (inv - (acc[p0x] >> 16) < size[p0x]) q -= g.twom - (int64_t)vol[p0x];
                }
                x = p0x;
            }
            contrib += (long long)g.deg[v] * q;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) contrib += __shfl_down_sync(kFull, contrib, o);
        if ((tid & 31) == 0 && contrib != 0) atomicAdd(&s_f, (unsigned long long)contrib);
        __syncthreads();
        if (tid == 0) task.f[t] = (int64_t)s_f;
    }
}

// ---- larger trees, in memory ------------------------------------------------
// Vertex word: target (low half); pops and the three flags above.
__device__ __forceinline__ uint64_t large_arrow(const PopTask &task, uint32_t sample, uint32_t v,
                                                uint32_t count) {
    const VRec r = load_rec(task.g.rec + v);
    const uint32_t k = bounded_draw_k(task.keys, task.seed, v, count, sample, kTagWalk,
                                      (uint32_t)r.deg);
    return (uint32_t)nbr_of(r, k, task.g.col);
}

constexpr int kFirstTrees = 4;  // trees for which a thread keeps a vertex's record
__global__ void __launch_bounds__(256) k_first_arrows(PopTask task, int64_t B, uint64_t *words) {
    const int64_t n = task.g.n;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const VRec r = load_rec(task.g.rec + v);
    const int64_t t0 = (int64_t)blockIdx.y * kFirstTrees;
    const int64_t t1 = t0 + kFirstTrees < B ? t0 + kFirstTrees : B;
    for (int64_t t = t0; t < t1; ++t) {
        // settled words are not followed: the root's target is its parent, -1
        uint64_t x = (uint64_t)kSettled << 32 |
                     (v == task.root ? 0xFFFFFFFFu : (uint32_t)task.root);
        if (v != task.root && v != task.fixed) {
            const uint32_t k = bounded_draw_k(task.keys, task.seed, (uint32_t)v, 0,
                                              (uint32_t)task.sids[t], kTagWalk, (uint32_t)r.deg);
            x = (uint32_t)nbr_of(r, k, task.g.col);
        }
        words[t * n + v] = x;
    }
}

// As led_cycle; kFirst: every vertex is active.
template <bool kFirst>
__device__ __forceinline__ int32_t led_cycle_large(uint64_t *word, int32_t a) {
    int32_t x = w_next(word[a]);
    int32_t saved = -1, len = 1;
    uint32_t met = 0, power = 1;
    for (;; ++len) {
        const uint64_t w = word[x];
        const uint32_t hi = (uint32_t)(w >> 32);
        if (kFirst || hi >= kSettled) {
            if (hi & kSettled) break;
            if (x <= a) return x == a ? len : 0;
            if (x == saved) return 0;
            if (++met == power) {
                saved = x;
                power <<= 1;
                met = 0;
            }
        }
        x = w_next(w);
    }
    x = a;
    for (uint64_t w = word[x]; !((w >> 32) & kSettled); w = word[x]) {
        word[x] = w | (uint64_t)kSettled << 32;
        x = w_next(w);
    }
    return 0;
}

__device__ __forceinline__ void list_cycle(const uint64_t *word, int32_t *list, uint32_t at,
                                           int32_t a) {
    int32_t x = a;
    do {
        list[at++] = x;
        x = w_next(word[x]);
    } while (x != a);
}

__global__ void __launch_bounds__(256) k_first_cycles(int64_t n, uint64_t *words, int32_t *lists,
                                                      unsigned long long *found) {
    const int64_t t = blockIdx.y;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t *word = words + t * n;
    if (v >= n || ((word[v] >> 32) & kSettled)) return;
    const int32_t len = led_cycle_large<true>(word, (int32_t)v);
    if (len)
        list_cycle(word, lists + t * n, (uint32_t)atomicAdd(found + t, (unsigned long long)len),
                   (int32_t)v);
}

template <int kThreads>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
    k_pop_rounds(PopTask task, uint64_t *words, int32_t *lists0, int32_t *lists1, int32_t *nexts,
                 const unsigned long long *found0) {
    const int64_t t = blockIdx.x, n = task.g.n;
    const uint32_t sample = (uint32_t)task.sids[t], tid = threadIdx.x;
    uint64_t *word = words + t * n;
    int32_t *list = lists0 + t * n, *fresh = lists1 + t * n, *next = nexts + t * n;
    __shared__ uint32_t s_count[2];
    uint32_t active = (uint32_t)found0[t];
    int64_t pops = 0;
    int end = 0;
    if (tid < 2) s_count[tid] = 0;
    for (int round = 0;; ++round) {
        pops += active;
        if (pops + n - task.placed > task.step_cap) {  // also of a first map that is a tree
            end = kErrStepLimit;
            break;
        }
        if (active == 0) break;
        __syncthreads();
        bool full = false;
        for (uint32_t i = tid; i < active; i += kThreads) {
            const int32_t v = list[i];
            const uint32_t c = ((uint32_t)(word[v] >> 32) & (kOnCycle - 1u)) + 1;
            word[v] = large_arrow(task, sample, (uint32_t)v, c) | (uint64_t)(c | kActive) << 32;
            full = full || c >= kWalkCountMask;
        }
        if (__syncthreads_or(full)) {
            end = kErrCountField;
            break;
        }
        if (active <= kHold * kThreads) {
            const uint64_t settled = (uint64_t)kSettled << 32;
            uint32_t len[kHold];
            for (int j = 0; j < kHold; ++j) {
                const uint32_t i = tid + j * kThreads;
                if (i >= active) break;
                const int32_t a = list[i];
                int32_t x = w_next(word[a]);
                uint64_t w = word[x];
                uint32_t l = 1;
                for (; w < settled; ++l) {
                    x = w_next(w);
                    w = word[x];
                }
                len[j] = l;
                next[a] = (w & settled) ? -1 : x;
            }
            __syncthreads();
            square_map<kThreads>(list, active, next);
            for (uint32_t i = tid; i < active; i += kThreads) {
                const int32_t h = next[list[i]];
                if (h >= 0) word[h] |= (uint64_t)kOnCycle << 32;
            }
            __syncthreads();
            for (int j = 0; j < kHold; ++j) {
                const uint32_t i = tid + j * kThreads;
                if (i >= active) break;
                int32_t x = list[i];
                uint64_t w = word[x];
                if ((w >> 32) & kOnCycle) {  // its piece of the cycle
                    uint32_t at = atomicAdd(&s_count[round & 1], len[j]);
                    do {
                        fresh[at++] = x;
                        x = w_next(w);
                        w = word[x];
                    } while (!((w >> 32) & kActive));
                } else if (next[x] < 0) {  // its piece of a path to the root
                    do {
                        word[x] = w | settled;
                        x = w_next(w);
                        w = word[x];
                    } while (w < settled);
                }
            }
        } else {
            for (uint32_t i = tid; i < active; i += kThreads) {
                const int32_t a = list[i];
                if ((word[a] >> 32) & kSettled) continue;
                const int32_t len = led_cycle_large<false>(word, a);
                if (len)
                    list_cycle(word, fresh, atomicAdd(&s_count[round & 1], (uint32_t)len), a);
            }
        }
        __syncthreads();
        for (uint32_t i = tid; i < active; i += kThreads)
            word[list[i]] &= ~((uint64_t)(kActive | kOnCycle) << 32);
        active = s_count[round & 1];
        if (tid == 0) s_count[(round + 1) & 1] = 0;
        int32_t *const swap = list;
        list = fresh;
        fresh = swap;
    }
    if (tid == 0) {
        if (end) atomicOr(task.err, (uint32_t)end);
        task.steps[t] = end ? -1 : pops + n - task.placed;
    }
}

// Parents of the finished maps, all trees of a wave in one run of `count` words.  It
// only reads the words: clearing them on the way for the traversal took 14 ms for
// 768 million of them, reading and then clearing takes 1.3 and 0.9.
__global__ void __launch_bounds__(256) k_take_parents(int64_t count, const uint64_t *words,
                                                      int32_t *par) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count;
         k += (int64_t)gridDim.x * blockDim.x)
        par[k] = w_next(words[k]);
}

constexpr int kMostDynamic = 224 * 1024;  // of 227 KB a block; the static part is small
static_assert(kc_host::pop_small_bytes(kc_host::kPopSmallMax) <= kMostDynamic &&
                  kc_host::pop_trees_bytes(kc_host::kPopContractMax) <= kMostDynamic &&
                  kc_host::pop_trees_bytes(kc_host::kPopTreesMax) <= kMostDynamic,
              "the largest trees fit a block");

// The kernel's shared memory is raised once per device, on its first call there.
template <int kThreads, bool kMulti, int kKind>
cudaError_t raise_shared() {
    static std::atomic<uint64_t> raised{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !((raised.load() >> dev) & 1u)) {
        e = cudaFuncSetAttribute(k_pop_small<kThreads, kMulti, kKind>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kMostDynamic);
        if (e != cudaSuccess) return e;
        if (dev < 64) raised.fetch_or((uint64_t)1 << dev);
    }
    return cudaSuccess;
}

template <int kThreads, bool kMulti, int kKind>
cudaError_t launch_small(const PopTask &one, const PopTask *tasks, const int2 *entry,
                         int64_t blocks, int64_t max_n, cudaStream_t s) {
    const size_t bytes =
        kKind == kFused ? kc_host::pop_small_bytes(max_n) : kc_host::pop_trees_bytes(max_n);
    const cudaError_t e = raise_shared<kThreads, kMulti, kKind>();
    if (e != cudaSuccess) return e;
    k_pop_small<kThreads, kMulti, kKind><<<(unsigned)blocks, kThreads, bytes, s>>>(one, tasks,
                                                                                   entry);
    return cudaGetLastError();
}

template <bool kMulti, int kKind>
cudaError_t launch_small_any(const PopTask &one, const PopTask *tasks, const int2 *entry,
                             int64_t blocks, int64_t max_n, cudaStream_t s) {
    if (blocks <= 0) return cudaSuccess;
    switch (kc_host::pop_small_threads(max_n)) {
        case 128: return launch_small<128, kMulti, kKind>(one, tasks, entry, blocks, max_n, s);
        case 256: return launch_small<256, kMulti, kKind>(one, tasks, entry, blocks, max_n, s);
        case 512: return launch_small<512, kMulti, kKind>(one, tasks, entry, blocks, max_n, s);
        default: return launch_small<1024, kMulti, kKind>(one, tasks, entry, blocks, max_n, s);
    }
}

}  // namespace

cudaError_t launch_pop_small(const PopTask &task, int64_t B, cudaStream_t s) {
    return launch_small_any<false, kFused>(task, nullptr, nullptr, B, task.g.n, s);
}

cudaError_t launch_pop_trees(const PopTask &task, int64_t B, cudaStream_t s) {
    return task.g.rec ? launch_small_any<false, kTrees>(task, nullptr, nullptr, B, task.g.n, s)
                      : launch_small_any<false, kTreesCsr>(task, nullptr, nullptr, B, task.g.n, s);
}

cudaError_t prepare_pop_trees_csr() {
    cudaError_t e = raise_shared<128, false, kTreesCsr>();
    if (e == cudaSuccess) e = raise_shared<256, false, kTreesCsr>();
    if (e == cudaSuccess) e = raise_shared<512, false, kTreesCsr>();
    if (e == cudaSuccess) e = raise_shared<1024, false, kTreesCsr>();
    return e;
}

cudaError_t launch_pop_small_multi(const PopTask *tasks, const int2 *entry, int64_t count,
                                   int64_t max_n, cudaStream_t s) {
    return launch_small_any<true, kFused>(PopTask{}, tasks, entry, count, max_n, s);
}

cudaError_t launch_pop_large(const PopTask &task, int64_t B, uint64_t *words, int32_t *lists0,
                             int32_t *lists1, int32_t *nexts, int64_t *found, int64_t num_sms,
                             cudaStream_t s) {
    const int64_t n = task.g.n;
    const cudaError_t e = cudaMemsetAsync(found, 0, sizeof(int64_t) * (size_t)B, s);
    if (e != cudaSuccess) return e;
    unsigned long long *count = reinterpret_cast<unsigned long long *>(found);
    const unsigned rows = (unsigned)((n + 255) / 256);
    k_first_arrows<<<dim3(rows, (unsigned)((B + kFirstTrees - 1) / kFirstTrees)), 256, 0, s>>>(
        task, B, words);
    k_first_cycles<<<dim3(rows, (unsigned)B), 256, 0, s>>>(n, words, lists0, count);
    if (B <= num_sms)
        k_pop_rounds<1024><<<(unsigned)B, 1024, 0, s>>>(task, words, lists0, lists1, nexts, count);
    else
        k_pop_rounds<256><<<(unsigned)B, 256, 0, s>>>(task, words, lists0, lists1, nexts, count);
    k_take_parents<<<(unsigned)std::min<int64_t>((B * n + 255) / 256, 64 * num_sms), 256, 0, s>>>(
        B * n, words, task.par);
    return cudaGetLastError();
}

}  // namespace kc
