// Wave planning for kc_sample (host side): how many trees a Wilson wave and a
// traversal sub-wave hold within a device-memory budget, and the workspace
// bytes a plan needs.
//
// Per tree of a Wilson wave: the walker words and the parent-first order
// (12 bytes a vertex).  Per tree of a traversal sub-wave: sizes, volumes and the
// DFN (16 bytes a vertex), the id-ordered sibling sums or preorder (4 more),
// and for the BIT evaluation of f the Fenwick array (8 more) -- its DFS stack is
// a separate allocation sized after the walk.  Low-eccentricity graphs (tau0
// scan) spend more time in the traversal than in the walk, so both get the same
// count; long-diameter graphs (BIT) spend most of it walking, which gets 70% of
// the budget by default (less when that would leave no room for one sub-wave
// tree).
//
// Plain C++ (no CUDA): the same header is compiled by the host tests.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>

namespace kc_host {

struct Plan {
    int64_t BW = 0;        // trees per Wilson wave
    int64_t BT = 0;        // trees per traversal sub-wave
    bool bit = false;
    int64_t stack_cap = 0; // BIT stack entries per tree
    bool canon = true;     // sub-wave buffers for the id-ordered DFN (aux array)
};

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Workspace bytes of a plan on an n-vertex graph (the layout carved from it).
inline size_t ws_bytes(int64_t n_vertices, const Plan &p) {
    const size_t n = (size_t)n_vertices;
    size_t b = 0;
    b += align256(sizeof(uint64_t) * n * p.BW);      // word
    b += align256(sizeof(int32_t) * n * p.BW);       // ord
    b += 3 * align256(sizeof(int64_t) * p.BW);       // steps, f, sids
    b += 2 * align256(sizeof(int32_t) * p.BW) + 256;  // hybrid hand-off: rs_q, rs_pos, done
    b += align256(sizeof(int32_t) * n * p.BT);       // size
    b += align256(sizeof(int64_t) * n * p.BT);       // vol
    b += align256(sizeof(int32_t) * n * p.BT);       // din
    if (p.bit || p.canon) b += align256(sizeof(int32_t) * n * p.BT);  // aux
    if (p.bit) b += align256(sizeof(int64_t) * (n + 1) * p.BT);  // bit
    return b;
}

// Wave sizes for ntrees trees within `budget` bytes (at least one tree each;
// max_in_flight > 0 caps the wave).  walker_share: the part of the budget the
// BIT variant gives to the Wilson wave (0.7; waves whose traversal streams
// through chunks of finished trees can give it more).
inline Plan plan_waves(int64_t n_vertices, int64_t ntrees, bool bit, bool canon, double budget,
                       int64_t max_in_flight, double walker_share = 0.7) {
    Plan p;
    p.bit = bit;
    p.canon = canon;
    const double n = (double)n_vertices;
    const double per_w = 12.0 * n + 64.0 + 8.0;
    const double per_t = (p.bit ? 28.0 : (canon ? 20.0 : 16.0)) * n + 64.0 +
                         (p.bit ? 16.0 * 4096.0 : 0.0);
    int64_t bw, bt;
    if (p.bit) {
        bw = (int64_t)std::floor(walker_share * budget / per_w);
        // leave room for at least one sub-wave tree
        bw = std::min<int64_t>(bw, (int64_t)std::floor((budget - per_t) / per_w));
        bw = std::max<int64_t>(1, std::min<int64_t>(bw, ntrees));
        if (max_in_flight > 0) bw = std::min(bw, max_in_flight);
        bw = std::min<int64_t>(bw, 1 << 20);
        bt = (int64_t)std::floor((budget - (double)bw * per_w) / per_t);
    } else {
        bw = (int64_t)std::floor(budget / (per_w + per_t));
        bw = std::max<int64_t>(1, std::min<int64_t>(bw, ntrees));
        if (max_in_flight > 0) bw = std::min(bw, max_in_flight);
        bw = std::min<int64_t>(bw, 1 << 20);
        bt = bw;
    }
    bt = std::max<int64_t>(1, std::min<int64_t>(bt, bw));
    bt = std::min<int64_t>(bt, 65535);
    p.BW = bw;
    p.BT = bt;
    p.stack_cap = p.bit ? 4096 : 0;
    return p;
}

// Trees a rejection wave draws so that it accepts `need` trees: need / rate
// plus three standard deviations of the accepted count, rate being the
// acceptance rate seen on the handle so far ((accepted + 1) / (drawn + 1),
// at least 1/64), or `hint` before any tree is seen.
inline int64_t reject_wave_size(int64_t need, int64_t drawn, int64_t accepted, double hint) {
    const double rate = drawn > 0 ? std::max(1.0 / 64.0, (double)(accepted + 1) /
                                                             (double)(drawn + 1))
                                  : hint;
    const double want = (double)need / rate;
    const double sd = std::sqrt(want * rate * (1.0 - rate)) / rate;
    return (int64_t)std::ceil(want + 3.0 * sd) + 8;
}

// Arrow queues of the one-walker kernels (k1_solo.cu): bits of a neighbour index
// in a graph of largest degree max_deg (at least 2), and how many arrows a queue of
// 32 bits holds behind the last one taken and before its end mark.  At most
// kMaxQueueBits bits leave room for one.
constexpr int kMaxQueueBits = 15;
constexpr int queue_bits(int64_t max_deg) {
    int b = 2;
    while (b < 63 && ((int64_t)1 << b) < max_deg) ++b;
    return b;
}
constexpr int queue_slots(int bits) { return (31 - bits) / bits; }

// Lanes per tree of those kernels for a wave of B trees: one tree per warp, which
// has the shortest chain per departure, unless the wave is a little too large for
// all of them to be resident (32 an SM) and two trees per warp make them so (48).
// 350x350 grid under a cap of 13 n departures, walk in ms for 32 / 16 / 8 lanes: 3044
// trees 260 / 362 / 523, 4522 trees 345 / 397 / 546, 5991 trees 482 / 430 / 575, 8929
// trees 628 / 742 / 620, 17672 trees 1133 / 1174 / 1204.  Without a cap, 32 / 16 lanes:
// grid 200x200, 5400 trees 256 / 272, 6000 trees 296 / 286, 7290 trees 301 / 309; random
// graph of 20000 vertices, 5400 trees 58 / 61, 6600 trees 67 / 62, 7290 trees 68 / 64, 7400
// trees 70 / 83; power-law graph of 20000, 4800 trees 26 / 32, 4880 trees 37 / 32, 7290
// trees 44 / 34, 7400 trees 44 / 51; K_300, 6000 trees 1.15 / 1.27.  The range pays from
// about 40 trees an SM on, on hubs in all of it.
inline int queue_group(int64_t B, int64_t num_sms) {
    const int64_t per_sm = (B + std::max<int64_t>(num_sms, 1) - 1) / std::max<int64_t>(num_sms, 1);
    return per_sm > 32 && per_sm <= 48 ? 16 : 32;
}

// Whether the LANE walker's wave of B trees runs those kernels, a warp or half a warp a
// tree, or (so many trees that lanes fill the GPU) a lane a tree.  The line, in trees an
// SM, depends on how even the walks are: about 145 to 205 on graphs of low diameter, 260
// and more on long-diameter ones, 180 there under a cap that ends long walks early.
// GB300, ms of a lane / a warp a tree: random graph of 300 vertices, 16000 trees 2.3 / 1.9,
// 128000 trees 7.2 / 13.3; of 2000, 32000 trees 25 / 25, 64000 trees 35 / 50; grid 10x10,
// 32000 trees 1.9 / 1.7, 256000 trees 6.7 / 12.0; grid 60x60, 32000 trees 109 / 68; grid
// 100x100 under a cap, 16000 accepted trees 162 / 149, 32000 trees 221 / 291.
inline bool queue_serves(int64_t B, int64_t num_sms, bool bit, bool reject) {
    return B < std::max<int64_t>(num_sms, 1) * (!bit ? 160 : (reject ? 184 : 320));
}

// Whether the retained trees that an ISM operation transforms, B of n vertices, are
// traversed by a warp a tree in a parent-first order (launch_prepare_from_parents,
// k2_traverse.cu) or by the order-free passes (k2_parents.cu), whose time is that of all
// vertices: the first where its warps fill the GPU.  GB300, tree part of an insertion and
// its deletion in ms, ordered / order-free: random graph of 2000 vertices, some 500 trees
// 5.6 / 5.1, 2000 trees 8.4 / 11.3, 5000 trees 18.4 / 25.2; of 16500, 500 trees 35 / 26,
// 2000 trees 87 / 83; of 60000, 500 trees 119 / 66; grid 100x100, 120 trees 18 / 12, 600
// trees 25.6 / 26.7, 4800 trees 100 / 144; grid 300x300, 120 trees 148 / 70, 600 trees
// 174 / 180.
inline bool transform_in_order(int64_t B, int64_t n, int64_t num_sms, bool bit) {
    return B >= 4 * num_sms + (bit ? 0 : n / 10);
}

// Cycle popping in shared memory (k_pop_small): its bytes for n vertices (two
// words, a volume and a 16-bit size each; vertex ids are 16 bits), the largest n
// (227 KB a block, less its static part) and the threads of a block.
constexpr size_t pop_small_bytes(int64_t n) { return (size_t)n * 12 + ((size_t)n * 2 + 3) / 4 * 4; }
constexpr int64_t kPopSmallMax = 16000;
// Trees without f hold 6 bytes a vertex there, past kPopContractMax 4.
constexpr int64_t kPopContractMax = 38000, kPopTreesMax = 56000;
constexpr size_t pop_trees_bytes(int64_t n) {
    return (size_t)n * (n <= kPopContractMax ? 6 : 4);
}
// Whether kc_wilson_noalloc pops its trees, a block each: while a block holds a tree and
// there are at most 128 of them a vertex.  Past that a lane per tree, of few
// departures each, fills the GPU better (GB300, ms of a lane per tree / popped, grid
// 6x6: 14600 trees 0.41 / 0.74, 233000 trees 1.2 / 8.6; random graph of 100 vertices:
// 10500 trees 0.34 / 0.29, 84000 trees 0.64 / 1.47; of 300: 28000 trees 1.7 / 1.2).
constexpr int64_t kPopTreesPerVertex = 128;
constexpr bool pop_noalloc(int64_t n, int64_t n_trees) {
    return n <= kPopTreesMax && n_trees <= kPopTreesPerVertex * n;
}
// How AUTO draws the trees of a low-diameter graph (against 32 walkers a tree and
// their traversal; GB300, ms):
//   up to kPopSmallMax vertices in shared memory, f included (random graph of 8000
//   vertices, 1000 trees 13.6 -> 6.3; of 15000 24.0 -> 12.4; power-law graph of 10000,
//   500 trees 5.3 -> 0.9);
//   past it in memory where the root is a hub, so that the walk to it, of about
//   2m / deg(root) departures, is short and the rounds touch few vertices (2 million
//   vertices, 384 trees 830 -> 140);
//   otherwise trees in shared memory while a block holds them.
enum : int { kPopNone = 0, kPopSmall = 1, kPopLarge = 2, kPopTrees = 3 };
inline int pop_kind(int64_t n, int64_t twom, int64_t root_deg) {
    if (n <= kPopSmallMax && twom < ((int64_t)1 << 32)) return kPopSmall;
    if (16 * (twom / std::max<int64_t>(root_deg, 1)) <= n) return kPopLarge;
    return n <= kPopContractMax ? kPopTrees : kPopNone;
}
// Threads of a block: most of a tree's time is a few long chains, so blocks stay small
// enough that an SM holds as many as its shared memory does.
inline int pop_small_threads(int64_t n) {
    return n <= 1024 ? 128 : (n <= 4096 ? 256 : (n <= 8192 ? 512 : 1024));
}

// Whether a row of the Laplacian product (k8_resistance.cu) is added up by 8 lanes, not by
// one thread: where some row is so long that the product would wait for its chain of
// loads.  The rows of random graphs of mean degree 20 and less are shorter, the hubs of
// power-law graphs longer (figures there).
constexpr bool spmv_by_lanes(int64_t max_deg) { return max_deg > 64; }

}  // namespace kc_host
