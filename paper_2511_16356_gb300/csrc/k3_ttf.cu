// f(tau) of Theorem 3 for every tree of a wave (Sec. 3.2).
//
// With p(x) the tau parent, p0(x) the tau0 parent and vol(x) = vol(Sub(tau, x)),
//   f(tau) = sum_{v != r} d(v) Q(v),
//   Q(v)   = sum over tau-ancestors x of v (x != r, x included when x = v) of
//              [p(x) = p0(x)]  [v in Sub(tau0, x)]    (2m - vol(x))      (forward)
//            - [p0(p(x)) = x]  [v in Sub(tau0, p(x))] (2m - vol(x))      (reverse)
// (Theorem 4 with the d(u) weight of Algorithm 1 and the reverse undo written as
// the negation of its add).  Two kernels evaluate it:
//
//  SCAN: for each v, walk up tau0 (at most its depth: ecc(r) for the BFS tree)
//        and test tau-ancestry with the DFN intervals of tau: O(n ecc) work, all
//        vertices of all trees in parallel.  Used when the depth is small (the
//        O(n Delta) bound of Thm 8).
//  BIT:  Algorithm 1's sum by a sweep over the preorder of tau with a Fenwick array
//        over the tau0 DFN (ttf_bit_sweep).  O(n log n) per tree, a warp a tree, 32
//        preorder positions per round.
// Both are templates: the batched instances take (graph, tree) entries and
// per-graph tables, so trees of many graphs share one launch.
#include <algorithm>

#include "kc_common.cuh"

namespace kc {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// kPar: parents from their arrays, else from the walker words
template <bool kMulti, bool kPar>
__global__ void __launch_bounds__(256) k_ttf_scan(GraphView g_in, WaveView w_in, MultiSub ms,
                                                  ParTrees trees) {
    GraphView g;
    WaveView w;
    int64_t t;
    if (!pick_tree<kMulti>(ms, g_in, w_in, blockIdx.y, g, w, t)) return;  // whole block
    const int64_t n = g.n;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t *__restrict__ word = w.word + wave_tree(w, t) * n;
    const int32_t *__restrict__ par = kPar ? trees.par + (trees.slot ? trees.slot[t] : t) * n
                                           : nullptr;
    const int32_t *__restrict__ din = w.din + t * n;
    const int32_t *__restrict__ size = w.size + t * n;
    const int64_t *__restrict__ vol = w.vol + t * n;
    const int32_t r = g.root;
    const int64_t twom = g.twom;
    long long contrib = 0;
    if (v < n && v != r) {
        const int32_t inv = din[v];
        long long q = 0;
        int32_t x = (int32_t)v;
        for (int it = 0; x != r && it <= g.ecc; ++it) {
            const int32_t p0x = g.p0[x];
            const int32_t px = kPar ? par[x] : w_next(word[x]);
            if (px == p0x) {
                const int32_t inx = din[x];
                if (inx <= inv && inv <= inx + size[x] - 1) q += twom - vol[x];
            } else if (p0x != r && (kPar ? par[p0x] : w_next(word[p0x])) == x) {
                const int32_t inw = din[p0x];
                if (inw <= inv && inv <= inw + size[p0x] - 1) q -= twom - vol[p0x];
            }
            x = p0x;
        }
        contrib = (long long)g.deg[v] * q;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) contrib += __shfl_down_sync(kFull, contrib, o);
    __shared__ long long part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = contrib;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long s = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += part[k];
        if (s != 0) atomicAdd((unsigned long long *)(w.f + wave_tree(w, t)), (unsigned long long)s);
    }
}

// The entry of tau-ancestor x (x != r, tau parent par) of Algorithm 1: kind 1 when
// p(x) = p0(x) (tau0-subtree of x, value 2m - vol(x)), kind 2 when p0(p(x)) = x
// (tau0-subtree of p(x), value vol(x) - 2m), 0 otherwise.
__device__ __forceinline__ int ttf_entry(const GraphView &g, int32_t x, int32_t par, int32_t r,
                                         int32_t twom, int64_t volx, int32_t &el, int32_t &er,
                                         int32_t &eval) {
    const int32_t vv = (int32_t)volx;
    if (g.p0[x] == par) {
        el = g.in0[x]; er = g.out0[x]; eval = twom - vv;
        return 1;
    }
    if (par != r && g.p0[par] == x) {
        el = g.in0[par]; er = g.out0[par]; eval = vv - twom;
        return 2;
    }
    return 0;
}

// Sum of a Fenwick array's first k entries, loads four at a time.
__device__ __forceinline__ int32_t bit_prefix(const int32_t *bit, uint32_t k) {
    int32_t s = 0;
    while (k) {
        int32_t x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[i] = k ? __ldcg(bit + k - 1) : 0;
            k &= k - 1;
        }
        s += x[0] + x[1] + x[2] + x[3];
    }
    return s;
}
__device__ __forceinline__ long long bit_range(const int32_t *bit, int32_t l, int32_t r) {
    return (long long)bit_prefix(bit, (uint32_t)r + 1u) - bit_prefix(bit, (uint32_t)l);
}

// Algorithm 1 the other way around.  Its sum over v of d(v) times the values of v's
// ancestors x whose tau0-interval [l, r] holds v equals, summed over x,
//   value(x) * D(x),  D(x) = sum of d(v) over v in Sub(tau, x) with in0(v) in [l, r],
// so the sweep over the preorder adds d(v) at point in0(v) and asks for the sum of
// [l, r] where Sub(tau, x) begins and where it ends: no range is added or undone.
// A warp takes 32 positions a round; within them D comes from the lanes, and
// only subtrees that reach past the round (kept on a stack) ask the Fenwick
// array, at the round's edges.  Sums of degrees fit 32 bits (2m < 2^31).
//
// What bounds it is the latency of a round: adding and undoing the ranges one
// position after the other took about 2000 cycles a position.  90000-vertex grid,
// 500 trees beside a running walk: 93 -> 30 ms; 6144 trees of small grids 5.8 -> 1.5.
//
// This lane's share of f over the preorder positions [lo, hi) of sub-wave tree t, on
// the zeroed array `bit` (n entries) and the stack `stk`, which holds sp entries
// {out, l, r, value}, the deepest on top, of subtrees that began before lo.
// ok = false on a stack overflow (the error bit is set).
__device__ __forceinline__ long long ttf_bit_sweep(const GraphView &g, const WaveView &w,
                                                   int64_t t, int32_t *bit, int4 *stk,
                                                   int64_t lo, int64_t hi, int64_t sp,
                                                   bool &ok) {
    const int lane = threadIdx.x & 31;
    const int64_t n = g.n;
    const int32_t r = g.root;
    const int32_t twom = (int32_t)g.twom;  // host guarantees 2m < 2^31 for this kernel
    const uint64_t *__restrict__ word = w.word + wave_tree(w, t) * n;
    const int32_t *__restrict__ size = w.size + t * n;
    const int64_t *__restrict__ vol = w.vol + t * n;
    const int32_t *__restrict__ pre = w.aux + t * n;
    const unsigned lt_mask = (1u << lane) - 1u;
    ok = true;

    long long facc = 0;     // this lane's share of f
    bool opened = false;    // its entry of the last round reached past it
    int32_t ol = 0, orr = 0, oval = 0;
    for (int64_t base = lo; base < hi; base += 32) {
        const int32_t last = (int32_t)((base + 32 < hi ? base + 32 : hi) - 1);
        const int64_t i = base + lane;
        const bool act = i < hi;
        int32_t v = -1, kind = 0, el = 0, er = 0, eval = 0, eout = 0, q = 0, dv = 0;
        if (act) {
            v = pre[i];
            if (v < 0 || v >= n) {  // preorder is a permutation; anything else is corrupt
                atomicOr(w.err, kErrBadTree);
                v = r;
            }
            q = g.in0[v];
            dv = g.deg[v];
            eout = (int32_t)i + size[v] - 1;
            if (v != r) kind = ttf_entry(g, v, w_next(word[v]), r, twom, vol[v], el, er, eval);
        }
        // ---- the array at the round's beginning: subtrees that the last round
        // opened, and those that this round ends
        if (opened) facc -= (long long)oval * bit_range(bit, ol, orr);
        int4 top = make_int4(0x7FFFFFFF, 0, 0, 0);
        if (sp - 1 - lane >= 0) top = stk[sp - 1 - lane];
        bool pop = top.x <= last;
        long long ended = pop ? bit_range(bit, top.y, top.z) : 0;
        // ---- the round's own points, for those and for the lanes' subtrees
        int32_t own = 0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const int32_t qj = __shfl_sync(kFull, q, j);
            const int32_t dj = __shfl_sync(kFull, dv, j);  // 0 past hi
            if (j >= lane && base + j <= eout && el <= qj && qj <= er) own += dj;
            if (base + j <= top.x && top.y <= qj && qj <= top.z) ended += dj;
        }
        if (kind) facc += (long long)eval * own;
        if (pop) facc += (long long)top.w * ended;
        unsigned popm = __ballot_sync(kFull, pop);  // outs ascend from the top down
        sp -= __popc(popm);
        while (popm == kFull && sp > 0) {  // more than a window of them
            top = make_int4(0x7FFFFFFF, 0, 0, 0);
            if (sp - 1 - lane >= 0) top = stk[sp - 1 - lane];
            pop = top.x <= last;
            ended = pop ? bit_range(bit, top.y, top.z) : 0;
            for (int j = 0; j < 32; ++j) {
                const int32_t qj = __shfl_sync(kFull, q, j);
                const int32_t dj = __shfl_sync(kFull, dv, j);
                if (base + j <= top.x && top.y <= qj && qj <= top.z) ended += dj;
            }
            if (pop) facc += (long long)top.w * ended;
            popm = __ballot_sync(kFull, pop);
            sp -= __popc(popm);
        }
        __syncwarp();  // every sum of the array above precedes the additions below
        if (act)
            for (int64_t k = (int64_t)q + 1; k <= n; k += k & -k) atomicAdd(bit + k - 1, dv);
        // ---- subtrees that reach past the round (at the end of a segment they
        // would be asked for twice on the same array: nothing is left)
        opened = kind && eout > last && base + 32 < hi;
        const unsigned open = __ballot_sync(kFull, opened);
        if (opened) {
            const int64_t slot = sp + __popc(open & lt_mask);
            if (slot < w.stack_cap) stk[slot] = make_int4(eout, el, er, eval);
            ol = el;
            orr = er;
            oval = eval;
        }
        sp += __popc(open);
        if (sp > w.stack_cap) {
            if (lane == 0) atomicOr(w.err, kErrBadTree);
            ok = false;
            return 0;
        }
        __threadfence_block();
        __syncwarp();
    }
    // subtrees that reach past hi
    for (int64_t e = lane; e < sp; e += 32) {
        const int4 x = stk[e];
        facc += (long long)x.w * bit_range(bit, x.y, x.z);
    }
    return facc;
}

template <bool kMulti>
__global__ void __launch_bounds__(128) k_ttf_bit(GraphView g_in, WaveView w_in, MultiSub ms) {
    const int lane = threadIdx.x & 31;
    GraphView g;
    WaveView w;
    int64_t t;
    if (!pick_tree<kMulti>(ms, g_in, w_in, ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                           g, w, t))
        return;
    const int64_t n = g.n;
    int32_t *bit = reinterpret_cast<int32_t *>(w.bit) + t * n;  // zeroed
    int4 *stk = reinterpret_cast<int4 *>(w.stack) + t * w.stack_cap;
    bool ok;
    long long facc = ttf_bit_sweep(g, w, t, bit, stk, 0, n, 0, ok);
    if (!ok) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) facc += __shfl_down_sync(kFull, facc, o);
    if (lane == 0) w.f[wave_tree(w, t)] = facc;
}

// The sweep over one preorder segment [lo, hi) of a tree per warp: D(x) is a sum
// over positions, so each segment adds its own points' share.  The subtrees that
// began before lo and reach into it are those of the strict tau-ancestors of u =
// pre[lo]; lane 0 collects them walking up the tau parents (deepest first) and the
// warp reverses them into stack order.  The segment's share of f is added to the
// tree's f, which the caller zeroed.
__global__ void __launch_bounds__(128) k_ttf_bit_seg(GraphView g, WaveView w,
                                                     const TtfSeg *__restrict__ segs,
                                                     int64_t nseg) {
    const int lane = threadIdx.x & 31;
    const int64_t si = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (si >= nseg) return;
    const TtfSeg sg = segs[si];
    const int64_t n = g.n;
    const int32_t r = g.root;
    const int32_t twom = (int32_t)g.twom;
    const int64_t t = sg.t;
    const uint64_t *__restrict__ word = w.word + wave_tree(w, t) * n;
    const int32_t *__restrict__ size = w.size + t * n;
    const int64_t *__restrict__ vol = w.vol + t * n;
    const int32_t *__restrict__ din = w.din + t * n;
    const int32_t *__restrict__ pre = w.aux + t * n;
    int4 *stk = sg.stk;
    int64_t sp = 0;
    if (sg.lo > 0) {
        long long cnt = 0;
        if (lane == 0) {
            const int32_t u = pre[sg.lo];
            int32_t x = (u >= 0 && u < n) ? w_next(word[u]) : -1;
            if (u < 0 || u >= n) cnt = -1;
            int64_t hops = 0;
            while (cnt >= 0 && x != r) {
                if (x < 0 || x >= n || ++hops > n) {
                    cnt = -1;
                    break;
                }
                const int32_t par = w_next(word[x]);
                if (par < 0 || par >= n) {  // only the root has no parent
                    cnt = -1;
                    break;
                }
                int32_t el = 0, er = 0, eval = 0;
                if (ttf_entry(g, x, par, r, twom, vol[x], el, er, eval)) {
                    if (cnt >= w.stack_cap) {
                        cnt = -1;
                        break;
                    }
                    stk[cnt++] = make_int4(din[x] + size[x] - 1, el, er, eval);
                }
                x = par;
            }
            if (cnt < 0) atomicOr(w.err, kErrBadTree);
        }
        cnt = __shfl_sync(kFull, cnt, 0);
        if (cnt < 0) return;
        __syncwarp();
        for (long long e = lane; e < cnt / 2; e += 32) {
            const int4 a = stk[e], b = stk[cnt - 1 - e];
            stk[e] = b;
            stk[cnt - 1 - e] = a;
        }
        __threadfence_block();
        __syncwarp();
        sp = cnt;
    }
    bool ok;
    int32_t *bit = reinterpret_cast<int32_t *>(sg.bit + 1);  // its first entry
    long long facc = ttf_bit_sweep(g, w, t, bit, stk, sg.lo, sg.hi, sp, ok);
    if (!ok) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) facc += __shfl_down_sync(kFull, facc, o);
    if (lane == 0 && facc != 0)
        atomicAdd((unsigned long long *)(w.f + wave_tree(w, t)), (unsigned long long)facc);
}

// zero every segment's Fenwick array
__global__ void k_zero_seg_bits(const TtfSeg *__restrict__ segs, int64_t nseg, int64_t n) {
    for (int64_t s = blockIdx.y; s < nseg; s += gridDim.y) {
        int32_t *b = reinterpret_cast<int32_t *>(segs[s].bit + 1);
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
             i += (int64_t)gridDim.x * blockDim.x)
            b[i] = 0;
    }
}

}  // namespace

cudaError_t launch_ttf_scan(const GraphView &g, WaveView w, cudaStream_t s) {
    if (!w.tmap) {  // with a tree map the caller has zeroed f for the whole wave
        cudaError_t e = cudaMemsetAsync(w.f, 0, sizeof(int64_t) * (size_t)w.B, s);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((unsigned)((g.n + 255) / 256), (unsigned)w.B);
    k_ttf_scan<false, false><<<grid, 256, 0, s>>>(g, w, MultiSub{}, ParTrees{});
    return cudaGetLastError();
}

cudaError_t launch_ttf_scan_parents(const GraphView &g, WaveView w, ParTrees trees,
                                    cudaStream_t s) {
    const cudaError_t e = cudaMemsetAsync(w.f, 0, sizeof(int64_t) * (size_t)w.B, s);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((g.n + 255) / 256), (unsigned)w.B);
    k_ttf_scan<false, true><<<grid, 256, 0, s>>>(g, w, MultiSub{}, trees);
    return cudaGetLastError();
}

cudaError_t launch_ttf_bit_seg(const GraphView &g, WaveView w, const TtfSeg *segs, int64_t nseg,
                              cudaStream_t s) {
    if (nseg <= 0) return cudaSuccess;
    const dim3 zgrid((unsigned)std::min<int64_t>((g.n + 255) / 256, 64),
                     (unsigned)std::min<int64_t>(nseg, 65535));
    k_zero_seg_bits<<<zgrid, 256, 0, s>>>(segs, nseg, g.n);
    k_ttf_bit_seg<<<(unsigned)((nseg * 32 + 127) / 128), 128, 0, s>>>(g, w, segs, nseg);
    return cudaGetLastError();
}

cudaError_t launch_ttf_bit(const GraphView &g, WaveView w, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(w.bit, 0, sizeof(int32_t) * (size_t)(w.B * g.n), s);
    if (e != cudaSuccess) return e;
    k_ttf_bit<false><<<(unsigned)((w.B * 32 + 127) / 128), 128, 0, s>>>(g, w, MultiSub{});
    return cudaGetLastError();
}

cudaError_t launch_ttf_scan_multi(const MultiSub &ms, int64_t max_n, cudaStream_t s) {
    for (int64_t r0 = 0; r0 < ms.count; r0 += 65535) {  // grid rows: at most 65535
        MultiSub part = ms;
        part.entry = ms.entry + r0;
        part.count = std::min<int64_t>(65535, ms.count - r0);
        dim3 grid((unsigned)((max_n + 255) / 256), (unsigned)part.count);
        k_ttf_scan<true, false><<<grid, 256, 0, s>>>(GraphView{}, WaveView{}, part, ParTrees{});
    }
    return cudaGetLastError();
}

cudaError_t launch_ttf_bit_multi(const MultiSub &ms, cudaStream_t s) {
    if (ms.count <= 0) return cudaSuccess;
    k_ttf_bit<true><<<(unsigned)((ms.count * 32 + 127) / 128), 128, 0, s>>>(GraphView{},
                                                                           WaveView{}, ms);
    return cudaGetLastError();
}

}  // namespace kc
