// Sample maintenance kernels (Sec. 4): BSM (Algorithm 2) and ISM (Algorithm 3).
//
//  - conditioned Wilson: walker words initialised with the edge (u, v) already
//    in the tree (u -> v, root v); the result is re-rooted at r;
//  - containment scan of the pool for an edge, Floyd selection of the trees to
//    replace or transform (Philox select stream);
//  - preparation of retained trees for the traversal passes: children lists,
//    then a warp-per-tree breadth-first pass giving depths and a parent-first
//    order;
//  - link-cut (ISM insertion) and cut-link (ISM deletion);
//  - weight rescaling with sums in a fixed order (bit-reproducible).
// The random choices follow the oracle's contract: tags select / link-cut /
// cut-link with counters (update seq, draw index or pool index, 0).
#include <algorithm>

#include "kc_common.cuh"

namespace kc {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

__global__ void k_edge_pre_init(int64_t n, int64_t B, int32_t u, int32_t v, uint64_t *word,
                                int32_t *ord) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= B) return;
    word[t * n + v] = w_make(-1, 0, true);
    word[t * n + u] = w_make(v, 1, true);
    ord[t * n] = v;
    ord[t * n + 1] = u;
}

// dst[slot[t]][x] = parent of x in wave tree t, from its words or (word null) its
// parent array
__global__ void k_words_to_slots(int64_t n, int64_t B, const uint64_t *word, const int32_t *par,
                                 const int64_t *slot, int32_t *pool_parents) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= B * n) return;
    const int64_t t = k / n, x = k - t * n;
    pool_parents[slot[t] * n + x] = word ? w_next(word[k]) : par[k];
}

// reverse the parent chain from r up to the old root `top` in each slot tree
__global__ void k_reroot_slots(int64_t n, int64_t B, const int64_t *slot, int32_t *pool_parents,
                               int32_t r, int32_t top, uint32_t *err) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= B || r == top) return;
    int32_t *p = pool_parents + slot[t] * n;
    int32_t prev = -1, cur = r;
    for (int64_t it = 0; it <= n; ++it) {
        const int32_t nxt = p[cur];
        p[cur] = prev;
        if (cur == top) return;
        if (nxt < 0 || nxt >= n) break;
        prev = cur;
        cur = nxt;
    }
    atomicOr(err, kErrBadTree);
}

__global__ void k_contains_edge(int64_t n, int64_t P, const int32_t *pool_parents, int32_t u,
                                int32_t v, uint8_t *flag) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    const int32_t *p = pool_parents + i * n;
    flag[i] = (p[u] == v || p[v] == u) ? 1 : 0;
}

// Floyd's sampling of k of [0, N) (one thread; `taken` zeroed, N bytes)
__global__ void k_select_floyd(uint64_t seed, uint32_t seq, int64_t N, int64_t k, uint8_t *taken,
                               int64_t *out) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    int64_t cnt = 0;
    for (int64_t j = N - k; j < N; ++j) {
        int64_t tt = (int64_t)bounded_draw(seed, seq, (uint32_t)cnt, 0, kTagSelect, (uint32_t)(j + 1));
        if (taken[tt]) tt = j;
        taken[tt] = 1;
        out[cnt++] = tt;
    }
}

// ---- preparation of parent arrays for the traversal passes ----------------
__global__ void k_gather_parents(int64_t n, int64_t B, const int32_t *pool_parents,
                                 const int64_t *slot, uint64_t *word, int32_t *cnt) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= B * n) return;
    const int64_t t = k / n;
    const int32_t p = pool_parents[slot[t] * n + (k - t * n)];
    word[k] = w_make(p, 0, false);
    if (p >= 0) atomicAdd(cnt + t * n + p, 1);
}

// exclusive scan of the child counts, warp per tree; off[t][n] is not stored
__global__ void __launch_bounds__(128) k_child_scan(int64_t n, int64_t B, const int32_t *cnt,
                                                    int32_t *off) {
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= B) return;
    int32_t carry = 0;
    for (int64_t base = 0; base < n; base += 32) {
        const int64_t x = base + lane;
        const int32_t c = x < n ? cnt[t * n + x] : 0;
        int32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        if (x < n) off[t * n + x] = carry + incl - c;
        carry += __shfl_sync(kFull, incl, 31);
    }
}

__global__ void k_child_scatter(int64_t n, int64_t B, const uint64_t *word, const int32_t *off,
                                int32_t *fill, int32_t *children) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= B * n) return;
    const int64_t t = k / n;
    const int32_t p = w_next(word[k]);
    if (p < 0) return;
    const int32_t pos = off[t * n + p] + atomicAdd(fill + t * n + p, 1);
    children[t * n + pos] = (int32_t)(k - t * n);
}

// Breadth-first order from the root (parent first) and depths, warp per tree.
__global__ void __launch_bounds__(128) k_bfs_order(int64_t n, int64_t B, int32_t root,
                                                   const int32_t *off, const int32_t *cnt,
                                                   const int32_t *children, uint64_t *word,
                                                   int32_t *ord, uint32_t *err,
                                                   int32_t *w_maxdepth) {
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= B) return;
    uint64_t *wd = word + t * n;
    int32_t *od = ord + t * n;
    const int32_t *ch = children + t * n;
    if (lane == 0) {
        od[0] = root;
        wd[root] = w_make(-1, 0, true);
    }
    __syncwarp();
    int64_t head = 0, tail = 1;
    while (head < tail) {
        const int64_t q = head + lane;
        int32_t v = -1, c = 0, o = 0;
        uint32_t dv = 0;
        if (q < tail) {  // entries written by other lanes: read at L2
            v = __ldcg(od + q);
            c = cnt[t * n + v];
            o = off[t * n + v];
            dv = w_count((uint64_t)__ldcg((const unsigned long long *)(wd + v)));
        }
        int32_t incl = c;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int32_t y = __shfl_up_sync(kFull, incl, s);
            if (lane >= s) incl += y;
        }
        const int32_t total = __shfl_sync(kFull, incl, 31);
        int64_t pos = tail + incl - c;
        for (int32_t j = 0; j < c; ++j) {
            const int32_t x = ch[o + j];
            if (pos < n) {
                __stcg(od + pos, x);
                __stcg((unsigned long long *)(wd + x), (unsigned long long)w_make(v, dv + 1, true));
            }
            ++pos;
        }
        if (c > 0) atomicMax(w_maxdepth, (int)dv + 1);
        const int64_t took = min((int64_t)32, tail - head);
        head += took;
        tail += total;
        __threadfence_block();
        __syncwarp();
        if (tail > n) {
            if (lane == 0) atomicOr(err, kErrBadTree);
            return;
        }
    }
    if (tail != n && lane == 0) atomicOr(err, kErrBadTree);
}

// ---- link-cut / cut-link ------------------------------------------------------
// Three steps over the selected trees: k_cut_choose (a thread a tree) finds the
// subtree that moves, k_cross_count counts the crossing edges in chunks of
// preorder positions with a block a chunk, and k_link_finish / k_cut_finish (a
// warp a tree) move the subtree.  The count is what the work is -- up to half the
// graph's edges a tree -- and with one warp a tree it took 28 (link-cut) and 51 ms
// (cut-link) for some 165 trees of 10^5 vertices.
constexpr int kCrossChunk = 256;  // preorder positions of a block

struct TransformIn {
    int64_t n;
    const int64_t *row_off;   // G'
    const int32_t *col;
    const int32_t *din;       // [B][n] DFN of the old tree
    const int32_t *size;      // [B][n]
    const int32_t *pre;       // [B][n] preorder -> vertex
    int32_t *scratch;         // [B][2n] int32: crossing edges of each chunk
    CutChoice *choice;        // [B]
    const int64_t *slot;      // [B] pool index of each tree
    int32_t *pool_parents;    // [P][n] the old trees, written in place
    double *factor;           // [B] d_old / d_new
    int32_t u, v;
    uint64_t seed;
    uint32_t seq;
    uint32_t *err;
};

__device__ __forceinline__ bool in_subtree(const int32_t *din, const int32_t *size, int32_t x,
                                           int32_t y) {  // y in Sub(x)
    return (uint32_t)(din[y] - din[x]) < (uint32_t)size[x];
}

// hops from a up to the lowest ancestor whose subtree holds b (returned in a)
__device__ int64_t climb_to(const int32_t *par, const int32_t *din, const int32_t *size, int32_t &a,
                            int32_t b, int64_t n) {
    int64_t d = 0;
    for (; d <= n && !in_subtree(din, size, a, b); ++d) a = par[a];
    return d;
}

__device__ int64_t hops_up(const int32_t *par, int32_t a, int32_t top, int64_t n) {
    int64_t d = 0;
    for (; d <= n && a != top; ++d) a = par[a];
    return d;
}

__device__ void reroot_chain(int32_t *p, int32_t x, int32_t top, int32_t attach, int64_t n,
                             uint32_t *err) {
    int32_t prev = attach, cur = x;
    for (int64_t it = 0; it <= n; ++it) {
        const int32_t nxt = p[cur];
        p[cur] = prev;
        if (cur == top) return;
        if (nxt < 0 || nxt >= n) break;
        prev = cur;
        cur = nxt;
    }
    atomicOr(err, kErrBadTree);
}

// The root x of the subtree that moves: link-cut draws an edge of the cycle that
// (u, v) closes (numbered from u up to the lowest common ancestor, then from v);
// cut-link has the end of (u, v) below the other.
__global__ void k_cut_choose(TransformIn a, int64_t B, bool insert) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= B) return;
    const int64_t n = a.n;
    const int32_t *par = a.pool_parents + a.slot[t] * n;
    const int32_t *din = a.din + t * n;
    const int32_t *size = a.size + t * n;
    CutChoice c;
    c.d_old = 0;
    if (insert) {
        int32_t top = a.u;
        const int64_t du = climb_to(par, din, size, top, a.v, n);
        const int64_t dv = hops_up(par, a.v, top, n);
        c.d_old = du + dv;
        int64_t k = (int64_t)bounded_draw(a.seed, a.seq, (uint32_t)a.slot[t], 0, kTagLinkCut,
                                          (uint32_t)c.d_old);
        c.side = k < du ? a.u : a.v;
        c.x = c.side;
        for (k = k < du ? k : k - du; k > 0; --k) c.x = par[c.x];
    } else {
        c.x = par[a.u] == a.v ? a.u : a.v;
        c.side = c.x == a.u ? a.v : a.u;  // the old parent
    }
    a.choice[t] = c;
}

// Crossing edges of the cut around Sub(x), a warp a vertex, a block a chunk of preorder
// positions.  Link-cut only needs their number, takes the positions of Sub(x) or of the
// rest, whichever are fewer, and leaves out the new edge (u, v) itself.  Cut-link takes
// those of Sub(x), whose chunks it searches for the edge that it draws: also where that is
// nearly all of the graph the chunks cost less than the warp per tree that tallied from
// the smaller side (root of degree 2 and one of its edges, deleted and inserted again:
// 2000 vertices and mean degree 12, pool of 20000 trees 16.3 -> 14.7 ms, power-law graph
// of 30000, 2000 trees 65 -> 17).
__global__ void __launch_bounds__(256) k_cross_count(TransformIn a, bool insert) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = a.n, t = blockIdx.y;
    const int32_t *__restrict__ din = a.din + t * n;
    const int32_t *__restrict__ pre = a.pre + t * n;
    const int32_t x = a.choice[t].x;
    const int32_t lo = din[x], sz = a.size[t * n + x];
    const bool inside = !insert || 2 * (int64_t)sz <= n;
    const int64_t span = inside ? (int64_t)sz : n - sz;
    __shared__ int32_t part[8];
    for (int64_t chunk = blockIdx.x; chunk * kCrossChunk < span; chunk += gridDim.x) {
        int32_t cross = 0;
        for (int i = warp; i < kCrossChunk; i += 8) {
            const int64_t k = chunk * kCrossChunk + i;
            if (k >= span) break;
            const int32_t y = pre[inside ? lo + k : (k < lo ? k : k + sz)];
            for (int64_t e = a.row_off[y] + lane; e < a.row_off[y + 1]; e += 32) {
                const int32_t z = a.col[e];
                if (((uint32_t)(din[z] - lo) < (uint32_t)sz) == inside) continue;
                if (insert && ((y == a.u && z == a.v) || (y == a.v && z == a.u))) continue;
                ++cross;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cross += __shfl_down_sync(kFull, cross, o);
        if (lane == 0) part[warp] = cross;
        __syncthreads();
        if (threadIdx.x == 0) {
            int32_t all = 0;
            for (int i = 0; i < 8; ++i) all += part[i];
            a.scratch[t * 2 * n + chunk] = all;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ long long warp_sum(long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

__global__ void __launch_bounds__(128) k_link_finish(TransformIn a, int64_t B) {
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= B) return;
    const int64_t n = a.n;
    const CutChoice c = a.choice[t];
    const int32_t sz = a.size[t * n + c.x];
    const int64_t span = 2 * (int64_t)sz <= n ? (int64_t)sz : n - sz;
    long long cross = 0;
    for (int64_t i = lane; i * kCrossChunk < span; i += 32) cross += a.scratch[t * 2 * n + i];
    cross = warp_sum(cross);
    if (lane == 0) {
        reroot_chain(a.pool_parents + a.slot[t] * n, c.side, c.x, c.side == a.u ? a.v : a.u, n,
                     a.err);
        a.factor[t] = cross > 0 ? (double)c.d_old / (double)cross : 0.0;
    }
}

// The k-th crossing edge in (preorder position of the inside end, outside end
// ascending) order: its chunk, then its position, then its place in the row.
__global__ void __launch_bounds__(128) k_cut_finish(TransformIn a, int64_t B) {
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= B) return;
    const int64_t n = a.n;
    int32_t *par = a.pool_parents + a.slot[t] * n;
    const int32_t *din = a.din + t * n;
    const int32_t *size = a.size + t * n;
    const int32_t *pre = a.pre + t * n;
    const int32_t *cnt = a.scratch + t * 2 * n;
    const CutChoice c = a.choice[t];
    const int32_t lo = din[c.x], sz = size[c.x];
    const int64_t chunks = ((int64_t)sz + kCrossChunk - 1) / kCrossChunk;
    long long cross = 0;
    for (int64_t i = lane; i < chunks; i += 32) cross += cnt[i];
    cross = warp_sum(cross);
    if (cross <= 0) {
        if (lane == 0) atomicOr(a.err, kErrBadTree);
        return;
    }
    long long k = 0;
    if (lane == 0)
        k = (long long)bounded_draw(a.seed, a.seq, (uint32_t)a.slot[t], 0, kTagCutLink,
                                    (uint32_t)cross);
    k = __shfl_sync(kFull, k, 0);
    int64_t chunk = -1;
    for (int64_t base = 0; base < chunks && chunk < 0; base += 32) {
        const int64_t i = base + lane;
        const long long mine = i < chunks ? (long long)cnt[i] : 0;
        long long incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const unsigned hit = __ballot_sync(kFull, k >= incl - mine && k < incl);
        if (hit) {
            const int src = __ffs(hit) - 1;
            chunk = base + src;
            k -= __shfl_sync(kFull, incl - mine, src);
        } else {
            k -= __shfl_sync(kFull, incl, 31);
        }
    }
    int32_t ia = -1, ob = -1;
    for (int64_t i = chunk * kCrossChunk; chunk >= 0 && i < sz && ia < 0; ++i) {
        if (i >= (chunk + 1) * kCrossChunk) break;
        const int32_t y = pre[lo + i];
        for (int64_t e0 = a.row_off[y]; e0 < a.row_off[y + 1]; e0 += 32) {
            int32_t z = -1;
            bool out = false;
            if (e0 + lane < a.row_off[y + 1]) {
                z = a.col[e0 + lane];
                out = (uint32_t)(din[z] - lo) >= (uint32_t)sz;
            }
            const unsigned m = __ballot_sync(kFull, out);
            if (k < __popc(m)) {
                const int src = __fns(m, 0, (int)k + 1);
                ia = y;
                ob = __shfl_sync(kFull, z, src);
                break;
            }
            k -= __popc(m);
        }
    }
    if (lane == 0) {
        if (ia < 0) {
            atomicOr(a.err, kErrBadTree);
            return;
        }
        int32_t top = ob;  // path ob .. the old parent, both outside Sub(x)
        const int64_t up = climb_to(par, din, size, top, c.side, n);
        const int64_t d_new = hops_up(par, ia, c.x, n) + 1 + up + hops_up(par, c.side, top, n);
        reroot_chain(par, ia, c.x, ob, n, a.err);
        a.factor[t] = (double)cross / (double)d_new;
    }
}

// ---- weights ----------------------------------------------------------------
// w[slot[j]] *= factor[j]
__global__ void k_scale_slots(double *w, const int64_t *slot, const double *factor, int64_t B) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < B) w[slot[j]] *= factor[j];
}

// sums over the pool in a fixed order: s[0] = sum over flagged, s[1] = unflagged
__global__ void __launch_bounds__(1024) k_weight_sums(const double *w, const uint8_t *flag,
                                                      int64_t P, double *s) {
    __shared__ double a[1024], b[1024];
    const int tid = threadIdx.x;
    double x = 0.0, y = 0.0;
    for (int64_t i = tid; i < P; i += blockDim.x) {
        if (flag[i]) x += w[i]; else y += w[i];
    }
    a[tid] = x;
    b[tid] = y;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (tid < h) {
            a[tid] += a[tid + h];
            b[tid] += b[tid + h];
        }
        __syncthreads();
    }
    if (tid == 0) {
        s[0] = a[0];
        s[1] = b[0];
    }
}

// flagged weights -> w / A * target_flagged, unflagged -> w / B * target_rest
// (a target < 0 leaves that group unchanged)
__global__ void k_weight_rescale(double *w, const uint8_t *flag, int64_t P, const double *s,
                                 double target_flagged, double target_rest) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    if (flag[i]) {
        if (target_flagged >= 0 && s[0] > 0) w[i] = w[i] / s[0] * target_flagged;
    } else {
        if (target_rest >= 0 && s[1] > 0) w[i] = w[i] / s[1] * target_rest;
    }
}

__global__ void k_scatter_results(const int64_t *slot, int64_t B, const int64_t *f,
                                  const int64_t *steps, const int64_t *sids, int64_t *pool_f,
                                  int64_t *pool_steps, int64_t *pool_sid) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= B) return;
    if (f) pool_f[slot[j]] = f[j];
    if (steps) pool_steps[slot[j]] = steps[j];
    if (sids) pool_sid[slot[j]] = sids[j];
}

inline unsigned blk(int64_t x, int t) { return (unsigned)((x + t - 1) / t); }

}  // namespace

cudaError_t launch_edge_pre_init(int64_t n, int64_t B, int32_t u, int32_t v, uint64_t *word,
                                 int32_t *ord, bool cleared, cudaStream_t s) {
    if (cleared) {
        cudaError_t e = cudaMemsetAsync(word, 0, sizeof(uint64_t) * (size_t)(B * n), s);
        if (e != cudaSuccess) return e;
    }
    k_edge_pre_init<<<blk(B, 128), 128, 0, s>>>(n, B, u, v, word, ord);
    return cudaGetLastError();
}

cudaError_t launch_words_to_slots(int64_t n, int64_t B, const uint64_t *word, const int32_t *par,
                                  const int64_t *slot, int32_t *pool_parents, int32_t r,
                                  int32_t top, uint32_t *err, cudaStream_t s) {
    k_words_to_slots<<<blk(B * n, 256), 256, 0, s>>>(n, B, word, par, slot, pool_parents);
    if (top >= 0) k_reroot_slots<<<blk(B, 128), 128, 0, s>>>(n, B, slot, pool_parents, r, top, err);
    return cudaGetLastError();
}

cudaError_t launch_contains_edge(int64_t n, int64_t P, const int32_t *pool_parents, int32_t u,
                                 int32_t v, uint8_t *flag, cudaStream_t s) {
    k_contains_edge<<<blk(P, 256), 256, 0, s>>>(n, P, pool_parents, u, v, flag);
    return cudaGetLastError();
}

cudaError_t launch_select(uint64_t seed, uint32_t seq, int64_t N, int64_t k, uint8_t *taken,
                          int64_t *out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(taken, 0, (size_t)N, s);
    if (e != cudaSuccess) return e;
    k_select_floyd<<<1, 1, 0, s>>>(seed, seq, N, k, taken, out);
    return cudaGetLastError();
}

// word/ord of wave trees from retained parent arrays: uses `cnt` (= size),
// `off` (= aux), `fill` (= din) and `children` (= vol reinterpreted) as scratch.
cudaError_t launch_prepare_from_parents(int64_t n, int64_t B, int32_t root,
                                        const int32_t *pool_parents, const int64_t *slot,
                                        WaveView w, cudaStream_t s) {
    const size_t per = sizeof(int32_t) * (size_t)(B * n);
    int32_t *cnt = w.size, *off = w.aux, *fill = w.din;
    int32_t *children = reinterpret_cast<int32_t *>(w.vol);
    cudaError_t e;
    if ((e = cudaMemsetAsync(cnt, 0, per, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(fill, 0, per, s)) != cudaSuccess) return e;
    k_gather_parents<<<blk(B * n, 256), 256, 0, s>>>(n, B, pool_parents, slot, w.word, cnt);
    k_child_scan<<<blk(B * 32, 128), 128, 0, s>>>(n, B, cnt, off);
    k_child_scatter<<<blk(B * n, 256), 256, 0, s>>>(n, B, w.word, off, fill, children);
    k_bfs_order<<<blk(B * 32, 128), 128, 0, s>>>(n, B, root, off, cnt, children, w.word, w.ord,
                                                 w.err, w.maxdepth);
    return cudaGetLastError();
}

cudaError_t launch_link_cut(const int64_t *row_off, const int32_t *col, WaveView w,
                            const int64_t *slot, int32_t *pool_parents, double *factor,
                            CutChoice *choice, int32_t u, int32_t v, uint64_t seed, uint32_t seq,
                            bool insert, cudaStream_t s) {
    TransformIn a;
    a.n = w.n;
    a.row_off = row_off;
    a.col = col;
    a.din = w.din;
    a.size = w.size;
    a.pre = w.aux;
    a.scratch = reinterpret_cast<int32_t *>(w.vol);  // 8n bytes per tree, unused here
    a.choice = choice;
    a.slot = slot;
    a.pool_parents = pool_parents;
    a.factor = factor;
    a.u = u;
    a.v = v;
    a.seed = seed;
    a.seq = seq;
    a.err = w.err;
    k_cut_choose<<<blk(w.B, 32), 32, 0, s>>>(a, w.B, insert);
    const dim3 grid((unsigned)std::min<int64_t>((w.n + kCrossChunk - 1) / kCrossChunk, 2048),
                    (unsigned)w.B);
    k_cross_count<<<grid, 256, 0, s>>>(a, insert);
    if (insert) k_link_finish<<<blk(w.B * 32, 128), 128, 0, s>>>(a, w.B);
    else k_cut_finish<<<blk(w.B * 32, 128), 128, 0, s>>>(a, w.B);
    return cudaGetLastError();
}

cudaError_t launch_scale_slots(double *w, const int64_t *slot, const double *factor, int64_t B,
                               cudaStream_t s) {
    k_scale_slots<<<blk(B, 256), 256, 0, s>>>(w, slot, factor, B);
    return cudaGetLastError();
}

cudaError_t launch_weight_rescale(double *w, const uint8_t *flag, int64_t P, double *sums,
                                  double target_flagged, double target_rest, cudaStream_t s) {
    k_weight_sums<<<1, 1024, 0, s>>>(w, flag, P, sums);
    k_weight_rescale<<<blk(P, 256), 256, 0, s>>>(w, flag, P, sums, target_flagged, target_rest);
    return cudaGetLastError();
}

cudaError_t launch_weight_sums(const double *w, const uint8_t *flag, int64_t P, double *sums,
                               cudaStream_t s) {
    k_weight_sums<<<1, 1024, 0, s>>>(w, flag, P, sums);
    return cudaGetLastError();
}

cudaError_t launch_scatter_results(const int64_t *slot, int64_t B, const int64_t *f,
                                   const int64_t *steps, const int64_t *sids, int64_t *pool_f,
                                   int64_t *pool_steps, int64_t *pool_sid, cudaStream_t s) {
    k_scatter_results<<<blk(B, 256), 256, 0, s>>>(slot, B, f, steps, sids, pool_f, pool_steps,
                                                  pool_sid);
    return cudaGetLastError();
}

}  // namespace kc
