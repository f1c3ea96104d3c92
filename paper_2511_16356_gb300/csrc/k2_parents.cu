// Traversal of trees given by their parent arrays, with no order of the vertices:
// subtree sizes, volumes and a preorder (Algorithm 1, "vol[u] <- the volume of
// Sub(tau_i, u)"; DFN of Sec. 3.2) by passes that are parallel over all vertices of
// all trees.
//
// The passes over a parent-first order (k2_traverse.cu) give a warp a tree and 32
// vertices a round trip, so a few hundred trees of 10^5 vertices and more leave
// the GPU idle.  Here every leaf starts a thread that reports its size and
// volume to its parent, and the last child to report goes on (k_par_up); a
// vertex's own word then holds its preorder relative to its parent, and all
// vertices jump to the root along those words at once (k_par_jump).
//
// Waves of deep trees (grids) stay with the passes over the order: a report and the last
// child's wait for it cost a chain of atomics per level, and beside a running walk
// those took 89 ms for the 4500 trees of a 350x350 grid where the ordered passes
// take 53, and slowed the walk by a tenth.  So do the trees of an ISM operation when
// they are many (kc_host::transform_in_order).  Fewer trees, and single ones, are
// traversed here on graphs of any depth (kc_get_tree of a 300x300 grid 97 -> 3.2 ms, of a
// 20x1000 grid 21 -> 1.8, of a path of 3000 vertices 4.8 -> 2.1).
//
// Word of a vertex (kc_host_par.h): until it reports, unreported children and sizes
// reported; then preorder offset and the ancestor it is relative to.  The second pair
// is read and written whole and holds at any time, so jumps need no rounds and no
// second buffer.  What bounds the passes
// is the rate of random 32-byte sectors.
//
// Measured (GB300, 100000-vertex power-law graph, 20 neighbours a vertex, pool of
// 1000 trees, 4 ISM operations of about 165 trees each): 743 -> 115 ms with the cut
// counts of k6_update.cu (about 60 with the later steps elsewhere); the warp-per-tree
// passes it replaces took 360 of the 743 (breadth-first order 176, child scan 25,
// top-down 56, sizes 80, siblings 21).
#include <algorithm>

#include <cuda/atomic>

#include "kc_common.cuh"
#include "kc_host_par.h"

namespace kc {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

__device__ __forceinline__ const int32_t *parents(const ParTrees &p, int64_t t, int64_t n) {
    return p.par + (p.slot ? p.slot[t] : t) * n;
}

__global__ void k_par_count(int64_t n, WaveView w, ParTrees trees) {
    const int64_t t = blockIdx.y;
    const int32_t *__restrict__ par = parents(trees, t, n);
    uint64_t *word = w.word + t * n;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = par[v];
        if (p >= 0 && p < n) atomicAdd((unsigned long long *)(word + p), 1ull << 32);
    }
}

// Only leaves start threads; a vertex's thread may come to it at any time, also after
// its tree is finished.
__global__ void k_par_up(GraphView g, WaveView w, ParTrees trees) {
    const int64_t n = g.n;
    const int64_t t = blockIdx.y;
    const int32_t *__restrict__ par = parents(trees, t, n);
    uint64_t *word = w.word + t * n;
    int32_t *size = w.size + t * n;
    int64_t *vol = w.vol + t * n;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        if (!kc_host::par_is_leaf(*(volatile unsigned long long *)(word + v), v, g.root)) continue;
        int32_t x = (int32_t)v, sx = 1;
        int64_t vx = (int64_t)g.deg[v];
        for (int64_t hop = 0;; ++hop) {
            const int32_t p = par[x];
            size[x] = sx;
            vol[x] = vx;
            if (p < 0 || p >= n || hop > n) {
                word[x] = kc_host::par_at(0, x);
                if (p >= n || hop > n || sx != n) atomicOr(w.err, kErrBadTree);
                break;
            }
            atomicAdd((unsigned long long *)(vol + p), (unsigned long long)vx);
            cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> acc(
                *reinterpret_cast<unsigned long long *>(word + p));
            const unsigned long long old =
                acc.fetch_add(kc_host::par_report(sx), cuda::memory_order_release);
            word[x] = kc_host::par_at((uint32_t)kc_host::par_sizes(old) + 1u, p);
            if (!kc_host::par_was_last(old)) break;  // siblings still to report
            cuda::atomic_thread_fence(cuda::memory_order_acquire, cuda::thread_scope_device);
            sx = 1 + kc_host::par_sizes(old) + sx;
            vx = (int64_t)g.deg[p] + *(volatile long long *)(vol + p);
            x = p;
        }
    }
}

// Offsets of the preorder that visits children in ascending id: a warp per vertex
// with children adds their sizes up along its row, which is ascending.  (eu, ev):
// an edge of the trees that the graph no longer holds (eu < 0: none).
__global__ void __launch_bounds__(256) k_par_sibling_rows(GraphView g, WaveView w,
                                                          ParTrees trees, int32_t eu,
                                                          int32_t ev) {
    const int lane = threadIdx.x & 31;
    const int64_t n = g.n;
    const int64_t t = blockIdx.y;
    const int32_t *__restrict__ par = parents(trees, t, n);
    const int32_t *__restrict__ size = w.size + t * n;
    uint64_t *word = w.word + t * n;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < n;
         p += warps) {
        if (size[p] == 1) continue;
        int32_t extra = -1;
        if (p == eu && par[ev] == eu) extra = ev;
        if (p == ev && par[eu] == ev) extra = eu;
        const int32_t extra_size = extra >= 0 ? size[extra] : 0;
        int32_t run = 0, below = 0;  // below: sizes of the children before `extra`
        for (int64_t e0 = g.row_off[p]; e0 < g.row_off[p + 1]; e0 += 32) {
            int32_t c = -1, sz = 0;
            if (e0 + lane < g.row_off[p + 1]) {
                c = g.col[e0 + lane];
                if (par[c] == p) sz = size[c];
            }
            int32_t incl = sz;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            if (sz) {
                const int32_t off = run + incl - sz + (extra >= 0 && extra < c ? extra_size : 0);
                word[c] = ((uint64_t)(uint32_t)off + 1ull) << 32 | (uint32_t)p;
                if (c < extra) below += sz;
            }
            run += __shfl_sync(kFull, incl, 31);
        }
        if (extra >= 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(kFull, below, o);
            if (lane == 0) word[extra] = ((uint64_t)(uint32_t)below + 1ull) << 32 | (uint32_t)p;
        }
    }
}

__global__ void k_par_jump(GraphView g, WaveView w, int want_pre) {
    const int64_t n = g.n;
    const int64_t t = blockIdx.y;
    volatile uint64_t *word = w.word + t * n;
    int32_t *din = w.din + t * n;
    int32_t *pre = w.aux + t * n;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        uint64_t p = word[v];
        bool bad = false;
        while ((int32_t)(uint32_t)p != g.root) {
            const uint32_t a = (uint32_t)p;
            if (a >= (uint64_t)n || (p >> 32) > (uint64_t)n) {  // not a tree rooted at g.root
                bad = true;
                break;
            }
            const uint64_t q = word[a];
            p = (((p >> 32) + (q >> 32)) << 32) | (uint32_t)q;
            word[v] = p;
        }
        const int32_t in = (int32_t)(p >> 32);
        if (bad || in >= n) {
            atomicOr(w.err, kErrBadTree);
            continue;
        }
        din[v] = in;
        if (want_pre) pre[in] = (int32_t)v;
    }
}

// the jumps that add up to the depths
__global__ void k_par_depth_init(GraphView g, WaveView w, ParTrees trees) {
    const int64_t n = g.n;
    const int64_t t = blockIdx.y;
    const int32_t *__restrict__ par = parents(trees, t, n);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        w.word[t * n + v] = v == g.root ? (uint64_t)(uint32_t)v
                                        : (1ull << 32 | (uint32_t)par[v]);
}

}  // namespace

cudaError_t launch_traverse_parents(const GraphView &g, WaveView w, ParTrees trees, bool by_id,
                                    int32_t eu, int32_t ev, bool want_preorder, cudaStream_t s,
                                    int *launches) {
    const size_t per = (size_t)(w.B * g.n);
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.word, 0, sizeof(uint64_t) * per, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.vol, 0, sizeof(int64_t) * per, s)) != cudaSuccess) return e;
    const dim3 grid((unsigned)std::min<int64_t>((g.n + 255) / 256, 4096), (unsigned)w.B);
    k_par_count<<<grid, 256, 0, s>>>(g.n, w, trees);
    k_par_up<<<grid, 256, 0, s>>>(g, w, trees);
    if (by_id) {
        const dim3 rows((unsigned)std::min<int64_t>((g.n + 7) / 8, 4096), (unsigned)w.B);
        k_par_sibling_rows<<<rows, 256, 0, s>>>(g, w, trees, eu, ev);
    }
    k_par_jump<<<grid, 256, 0, s>>>(g, w, want_preorder ? 1 : 0);
    if (launches) *launches += by_id ? 4 : 3;
    return cudaGetLastError();
}

cudaError_t launch_depths_parents(const GraphView &g, WaveView w, ParTrees trees,
                                  cudaStream_t s) {
    const dim3 grid((unsigned)std::min<int64_t>((g.n + 255) / 256, 4096), (unsigned)w.B);
    k_par_depth_init<<<grid, 256, 0, s>>>(g, w, trees);
    k_par_jump<<<grid, 256, 0, s>>>(g, w, 0);
    return cudaGetLastError();
}

}  // namespace kc
