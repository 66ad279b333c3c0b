// tree4.cu -- the traversal tree: a binary tree of the scene's leaves built by
// PLOC (Meister and Bittner 2018, "Parallel Locally-Ordered Clustering for
// Bounding Volume Hierarchy Construction"), collapsed into 4-wide nodes.
//
// PLOC starts from the leaves in Morton order (the LBVH sort) and repeats:
//   1. every cluster finds the cluster within +-kRadius positions whose
//      merged box has the smallest surface area (ties: the nearer position,
//      then the partner i ^ 1, so runs of equal boxes pair up);
//   2. mutual nearest neighbours merge into a new internal node, which takes
//      the lower position; the other position is dropped;
//   3. the cluster array is compacted (positions and node numbers from prefix
//      sums, no atomics, so the tree is deterministic).
// The pair of mutual neighbours with the smallest distance (lowest position on
// ties) always exists, so every round merges at least once.  A round keeps
// about 82 % of the clusters: 1.07 M leaves take some 70 rounds.
//
// A round is two launches (pair, merge) whose cluster count lives on the
// device, so the host enqueues all the rounds it expects without waiting, and
// once kTail clusters are left one block does the remaining rounds in shared
// memory.  (Twelve launches and a host wait to a round made clustering the
// larger part of a build: 1.07 M triangles and their first cast took 6.6 ms,
// now 1.6 ms, of which the rounds are about 0.4.)
//
// The tree is then collapsed two levels at a time: every internal node at even
// depth becomes a 4-wide node whose children are its children, internal
// children replaced by their own two children.  All boxes are exact FP32
// unions of the triangles' boxes.
#include "vafr_internal.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace vafr {
namespace {

constexpr int kRadius = 8;
constexpr int kRoundThreads = 512;
constexpr int kTile = kRoundThreads - 3 * kRadius;   // clusters per block of a round
constexpr int kTail = 2048;         // clusters that one block finishes
constexpr int kTailThreads = 1024;
constexpr int kMaxRounds = 100000;
constexpr int kScanBlocks = 4096;   // above: the blocks' counts get a scan of their own
constexpr int kThreads = 256;
constexpr int kHeadThreads = 1024;

inline int blocks_for(long long n, int tpb) { return (int)((n + tpb - 1) / tpb); }

// ---- PLOC ---------------------------------------------------------------------------
// A cluster or binary node is two float4: (lo.xyz, a), (hi.xyz, b).  Clusters: a
// = reference (>= 0 node, < 0 leaf ~k).  Nodes: (a, b) = the two children.
// Node ids are in order of creation, so the root is the last.

// State between rounds: clusters left, nodes made, the array that holds the
// clusters (0 or 1), and whether the last round merged nothing.
struct PlocState {
    int m, nodes, buf, stuck;
};

__device__ __forceinline__ float half_area(float4 lo, float4 hi) {
    const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return fmaf(dx, dy, fmaf(dy, dz, dz * dx));
}

// Merged areas of the cluster at position i of m and its kRadius successors,
// whose boxes are lo[0 .. kRadius], hi[..]; infinite past the end.  A pair's
// area is computed once, for the earlier of the two (which halves the box
// loads from shared memory that bounded a round).
__device__ __forceinline__ void pair_costs(const float4* lo, const float4* hi, int i, int m, float cost[kRadius]) {
    const float4 a = lo[0], A = hi[0];
#pragma unroll
    for (int d = 1; d <= kRadius; ++d) {
        cost[d - 1] = INFINITY;
        if (i + d < m) {
            const float4 b = lo[d], B = hi[d];
            cost[d - 1] = half_area(make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z), 0.0f),
                                    make_float4(fmaxf(A.x, B.x), fmaxf(A.y, B.y), fmaxf(A.z, B.z), 0.0f));
        }
    }
}

// Offset of the nearest neighbour of the cluster at position i: fore(d), back(d)
// are its costs with the clusters d positions on and before; 0: none.
// Equal costs (identical boxes, e.g. duplicated geometry) go to the nearer
// position, then to the partner i ^ 1: a run of equal boxes then pairs up
// as (0,1) (2,3) ... in every round and halves, where "lower position
// first" would merge one pair per round and chain the tree.  Trying the
// offsets in that order makes it a plain minimum.
template <class F, class B>
__device__ __forceinline__ int nearest(int i, F&& fore, B&& back) {
    float best = INFINITY;
    int bd = 0;
    auto attempt = [&](float c, int d) {
        if (c < best) {
            best = c;
            bd = d;
        }
    };
    const float f1 = fore(1), b1 = back(1);
    const bool odd = i & 1;
    attempt(odd ? b1 : f1, odd ? -1 : 1);
    attempt(odd ? f1 : b1, odd ? 1 : -1);
#pragma unroll
    for (int d = 2; d <= kRadius; ++d) {
        attempt(back(d), -d);
        attempt(fore(d), d);
    }
    return bd;
}

// What becomes of the cluster whose nearest neighbour is d away and has its
// own at back: 0 dropped (its partner takes it), 1 kept, 1 + d merged with the
// partner d positions on.
__device__ __forceinline__ int fate(int d, int back) {
    if (d == 0 || back != -d) return 1;
    return d < 0 ? 0 : 1 + d;
}

struct Ploc {
    float4 *clusters0, *clusters1;
    float4* nodes;          // binary nodes, two float4 each
    int32_t* parent;        // of each binary node
    unsigned char* fates;   // of each cluster
    unsigned* counts;       // per block: clusters kept | merged << 16, or their exclusive prefixes
    PlocState* state;       // [2], used alternately
};

// Merged pair (a, A), (b, B): node id, its record, its children's parent.
__device__ __forceinline__ void make_node(const Ploc& p, int id, float4 a, float4 A, float4 b, float4 B, float4& lo,
                                          float4& hi) {
    lo = make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z), a.w);
    hi = make_float4(fmaxf(A.x, B.x), fmaxf(A.y, B.y), fmaxf(A.z, B.z), b.w);
    p.nodes[2ll * id] = lo;
    p.nodes[2ll * id + 1] = hi;
    const int l = __float_as_int(a.w), r = __float_as_int(b.w);
    if (l >= 0) p.parent[l] = id;
    if (r >= 0) p.parent[r] = id;
    lo.w = __int_as_float(id);
}

// First launch of a round: each cluster's fate and each tile's counts.  A
// thread takes one position from 2 kRadius before the tile on (the clusters'
// neighbours' neighbours decide with it).  Blocks stride over the tiles, so
// the grid only has to be about right: the host shrinks it by the expected
// share from round to round (with a block for every tile of the first round,
// starting 2,089 mostly idle blocks took 9 us of each of the 64 launches).
__global__ void __launch_bounds__(kRoundThreads) k_ploc_pair(const Ploc p, int par) {
    constexpr int R = kRadius, T = kRoundThreads;
    __shared__ float4 slo[T + R], shi[T + R];
    __shared__ float scost[R][T];
    __shared__ signed char near[T];
    after_previous();
    const PlocState st = p.state[par];
    if (st.m <= kTail || st.stuck) return;
    const float4* cl = st.buf ? p.clusters1 : p.clusters0;
    const int tiles = (st.m + kTile - 1) / kTile;
    const int t = threadIdx.x;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int i = tile * kTile - 2 * R + t;   // may be negative: then it has no box
        for (int k = t; k < T + R; k += T) {
            const int j = i - t + k;
            if (j >= 0 && j < st.m) {
                slo[k] = cl[2ll * j];
                shi[k] = cl[2ll * j + 1];
            }
        }
        __syncthreads();
        float cost[R];
        pair_costs(slo + t, shi + t, i >= 0 ? i : st.m, st.m, cost);
#pragma unroll
        for (int d = 0; d < R; ++d) scost[d][t] = cost[d];
        __syncthreads();
        int d = 0;
        if (t >= R)
            d = nearest(i, [&](int q) { return cost[q - 1]; }, [&](int q) { return scost[q - 1][t - q]; });
        near[t] = (signed char)d;
        __syncthreads();
        int f = 0;
        if (t >= 2 * R && t < T - R && i < st.m) {
            f = fate(d, near[t + d]);
            p.fates[i] = (unsigned char)f;
        }
        const int kept = __syncthreads_count(f > 0), merged = __syncthreads_count(f > 1);
        if (t == 0) p.counts[tile] = (unsigned)kept | (unsigned)merged << 16;
    }
}

// Sum over the block of (kept, merged), both below 2^31, in two words.
__device__ __forceinline__ int2 block_sum(int2 v, int2* warp_sum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v.x = __reduce_add_sync(0xffffffffu, v.x);
    v.y = __reduce_add_sync(0xffffffffu, v.y);
    if (lane == 0) warp_sum[warp] = v;
    __syncthreads();
    int2 t = make_int2(0, 0);
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        t.x += warp_sum[w].x;
        t.y += warp_sum[w].y;
    }
    __syncthreads();
    return t;
}

// Second launch of a round: the compacted clusters and the new nodes.  A
// block sums the counts before its tiles itself (at 1.07 M clusters 4 MB of L2
// reads in all); k_ploc_scan does it where there are more than kScanBlocks.
__global__ void __launch_bounds__(kRoundThreads) k_ploc_merge(const Ploc p, int par, const int2* scanned) {
    __shared__ int2 warp_sum[kRoundThreads / 32];
    after_previous();
    const PlocState st = p.state[par];
    if (st.m <= kTail || st.stuck) {
        if (blockIdx.x == 0 && threadIdx.x == 0) p.state[par ^ 1] = st;
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int tiles = (st.m + kTile - 1) / kTile;
    int2 before = make_int2(0, 0);
    int summed = 0;   // tiles that `before` counts
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (scanned) {
            before = scanned[tile];
        } else {
            int2 c = make_int2(0, 0);
            for (int k = summed + (int)threadIdx.x; k < tile; k += kRoundThreads) {
                const unsigned v = p.counts[k];
                c.x += (int)(v & 0xffffu);
                c.y += (int)(v >> 16);
            }
            c = block_sum(c, warp_sum);
            before.x += c.x;
            before.y += c.y;
            summed = tile;
        }
        const int i = tile * kTile + (int)threadIdx.x;
        const int f = threadIdx.x < kTile && i < st.m ? (int)p.fates[i] : 0;
        const unsigned kept = __ballot_sync(0xffffffffu, f > 0), merged = __ballot_sync(0xffffffffu, f > 1);
        if (lane == 0) warp_sum[warp] = make_int2(__popc(kept), __popc(merged));
        __syncthreads();
        int2 in = make_int2(0, 0), all = make_int2(0, 0);
#pragma unroll
        for (int w = 0; w < kRoundThreads / 32; ++w) {
            const int2 c = warp_sum[w];
            if (w < warp) { in.x += c.x; in.y += c.y; }
            all.x += c.x;
            all.y += c.y;
        }
        if (f > 0) {
            const float4* cl = st.buf ? p.clusters1 : p.clusters0;
            float4* out = (st.buf ? p.clusters0 : p.clusters1) + 2ll * (before.x + in.x + __popc(kept & lt));
            float4 lo = cl[2ll * i], hi = cl[2ll * i + 1];
            if (f > 1) {
                const long long j = i + f - 1;
                make_node(p, st.nodes + before.y + in.y + __popc(merged & lt), lo, hi, cl[2 * j], cl[2 * j + 1], lo,
                          hi);
            }
            out[0] = lo;
            out[1] = hi;
        }
        if (threadIdx.x == 0 && tile == tiles - 1) {
            const int made = before.y + all.y;
            PlocState nx;
            nx.m = before.x + all.x;
            nx.nodes = st.nodes + made;
            nx.buf = st.buf ^ 1;
            nx.stuck = made <= 0 || nx.m != st.m - made;
            p.state[par ^ 1] = nx;
        }
        __syncthreads();   // warp_sum is used again
    }
}

// Exclusive prefixes of the blocks' counts, by one block.
__global__ void __launch_bounds__(1024) k_ploc_scan(const Ploc p, int par, int2* scanned) {
    __shared__ int2 warp_sum[32];
    after_previous();
    const PlocState st = p.state[par];
    if (st.m <= kTail || st.stuck) return;
    const int nb = (st.m + kTile - 1) / kTile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int2 carry = make_int2(0, 0);
    for (int base = 0; base < nb; base += 1024) {
        const int k = base + (int)threadIdx.x;
        const unsigned c = k < nb ? p.counts[k] : 0u;
        const int2 x = make_int2((int)(c & 0xffffu), (int)(c >> 16));
        int2 incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int yx = __shfl_up_sync(0xffffffffu, incl.x, o), yy = __shfl_up_sync(0xffffffffu, incl.y, o);
            if (lane >= o) { incl.x += yx; incl.y += yy; }
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        int2 in = make_int2(0, 0), all = make_int2(0, 0);
        for (int w = 0; w < 32; ++w) {
            const int2 v = warp_sum[w];
            if (w < warp) { in.x += v.x; in.y += v.y; }
            all.x += v.x;
            all.y += v.y;
        }
        if (k < nb) scanned[k] = make_int2(carry.x + in.x + incl.x - x.x, carry.y + in.y + incl.y - x.y);
        carry.x += all.x;
        carry.y += all.y;
        __syncthreads();
    }
}

// The last rounds, kTail clusters or fewer, by one block in shared memory:
// 1,024 threads down to 256 clusters, then 256 threads down to 32, then one
// warp (27 of the 37 rounds from 2,048 clusters on have 256 or fewer, and a
// round is then mostly its barriers).
struct TailShared {
    float4 lo[kTail], hi[kTail];
    float cost[kRadius][kTail];
    signed char near[kTail];
    int2 group[kTail / 32];   // per 32 consecutive positions: kept, merged; then their exclusive prefixes
    int2 total;
};

template <int T>
__device__ __forceinline__ void tail_sync() {
    if (T == 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
}

// Rounds by the block's first T threads, ITEMS clusters each, until `stop` or
// fewer are left.
template <int T, int ITEMS>
__device__ __forceinline__ void tail_rounds(const Ploc& p, TailShared& sh, int stop, int& m, int& nodes, bool& stuck) {
    static_assert(ITEMS == 1 || T * ITEMS / 32 == 32 * ITEMS, "a lane of the prefix sum takes ITEMS groups");
    constexpr int GROUPS = T * ITEMS / 32;
    const int t = threadIdx.x, lane = t & 31;
    const unsigned lt = (1u << lane) - 1u;
    while (m > stop && !stuck) {
        float cost[ITEMS][kRadius];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = t + k * T;
            if (i < m) {
                pair_costs(sh.lo + i, sh.hi + i, i, m, cost[k]);
#pragma unroll
                for (int d = 0; d < kRadius; ++d) sh.cost[d][i] = cost[k][d];
            }
        }
        tail_sync<T>();
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = t + k * T;
            if (i < m)
                sh.near[i] = (signed char)nearest(
                    i, [&](int q) { return cost[k][q - 1]; },
                    [&](int q) { return i >= q ? sh.cost[q - 1][i - q] : INFINITY; });
        }
        tail_sync<T>();
        int f[ITEMS];
        unsigned kept[ITEMS], merged[ITEMS];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = t + k * T;
            f[k] = 0;
            if (i < m) {
                const int d = sh.near[i];
                f[k] = fate(d, sh.near[i + d]);
            }
            kept[k] = __ballot_sync(0xffffffffu, f[k] > 0);
            merged[k] = __ballot_sync(0xffffffffu, f[k] > 1);
            if (lane == 0) sh.group[i >> 5] = make_int2(__popc(kept[k]), __popc(merged[k]));
        }
        tail_sync<T>();
        if (t < 32) {
            constexpr int PER = GROUPS > 32 ? GROUPS / 32 : 1;   // consecutive groups to a lane
            int2 x[PER], run = make_int2(0, 0);
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                x[k] = PER * t + k < GROUPS ? sh.group[PER * t + k] : make_int2(0, 0);
                run.x += x[k].x;
                run.y += x[k].y;
            }
            int2 incl = run;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int yx = __shfl_up_sync(0xffffffffu, incl.x, o), yy = __shfl_up_sync(0xffffffffu, incl.y, o);
                if (lane >= o) { incl.x += yx; incl.y += yy; }
            }
            if (t == 31) sh.total = incl;
            int2 pre = make_int2(incl.x - run.x, incl.y - run.y);
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                if (PER * t + k < GROUPS) sh.group[PER * t + k] = pre;
                pre.x += x[k].x;
                pre.y += x[k].y;
            }
        }
        tail_sync<T>();
        float4 lo[ITEMS], hi[ITEMS];
        int to[ITEMS];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = t + k * T;
            if (f[k] > 0) {
                const int2 pre = sh.group[i >> 5];
                to[k] = pre.x + __popc(kept[k] & lt);
                lo[k] = sh.lo[i];
                hi[k] = sh.hi[i];
                if (f[k] > 1) {
                    const int j = i + f[k] - 1;
                    make_node(p, nodes + pre.y + __popc(merged[k] & lt), lo[k], hi[k], sh.lo[j], sh.hi[j], lo[k], hi[k]);
                }
            }
        }
        const int2 total = sh.total;
        tail_sync<T>();
#pragma unroll
        for (int k = 0; k < ITEMS; ++k)
            if (f[k] > 0) {
                sh.lo[to[k]] = lo[k];
                sh.hi[to[k]] = hi[k];
            }
        tail_sync<T>();
        stuck = total.y <= 0 || total.x != m - total.y;
        if (!stuck) {
            m = total.x;
            nodes += total.y;
        }
    }
}

__global__ void __launch_bounds__(kTailThreads) k_ploc_tail(const Ploc p, int par) {
    extern __shared__ unsigned char raw[];
    TailShared& sh = *reinterpret_cast<TailShared*>(raw);
    after_previous();
    PlocState st = p.state[par];
    if (st.m > kTail || st.stuck) return;   // the host looks at the state
    const float4* cl = st.buf ? p.clusters1 : p.clusters0;
    for (int i = threadIdx.x; i < st.m; i += kTailThreads) {
        sh.lo[i] = cl[2 * i];
        sh.hi[i] = cl[2 * i + 1];
    }
    __syncthreads();
    bool stuck = false;
    tail_rounds<kTailThreads, kTail / kTailThreads>(p, sh, 256, st.m, st.nodes, stuck);
    if (threadIdx.x >= 256) return;
    tail_rounds<256, 1>(p, sh, 32, st.m, st.nodes, stuck);
    if (threadIdx.x >= 32) return;
    tail_rounds<32, 1>(p, sh, 1, st.m, st.nodes, stuck);
    if (threadIdx.x == 0) {
        st.stuck = stuck;
        p.state[par] = st;
    }
}

__global__ void k_ploc_start(PlocState* state, int n) {
    PlocState s;
    s.m = n;
    s.nodes = 0;
    s.buf = 0;
    s.stuck = 0;
    state[0] = s;
}

// ---- collapse to 4-wide -------------------------------------------------------------
// Node ids from the root on: node id n_inner - 1 - i is number i below.

__device__ __forceinline__ int2 children2(const float4* __restrict__ nodes, int id) {
    return make_int2(__float_as_int(nodes[2ll * id].w), __float_as_int(nodes[2ll * id + 1].w));
}

// The 4-wide children of head id: its binary children that are leaves and the
// two children of each internal one (heads, at the next even depth, or
// leaves).  Internal children come first (ni of them), then the leaves: m in
// all.  Each head's internal children get consecutive 4-wide indices, so the
// child in slot q < ni is the slot-0 child + q.
__device__ __forceinline__ void children4(const float4* __restrict__ nodes, int id, int ref[4], int& m, int& ni) {
    const int2 c = children2(nodes, id);
    const bool lx = c.x < 0, ly = c.y < 0;
    const int2 g = lx ? make_int2(c.x, kEmptyRef) : children2(nodes, c.x);
    const int2 h = ly ? make_int2(c.y, kEmptyRef) : children2(nodes, c.y);
    const int in[4] = {g.x, g.y, h.x, h.y};
    m = 4 - (lx ? 1 : 0) - (ly ? 1 : 0);
    ni = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) ni += in[q] >= 0 ? 1 : 0;
    int at = 0, leaf = ni;
    ref[0] = ref[1] = ref[2] = ref[3] = kEmptyRef;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (in[q] == kEmptyRef) continue;
        const int to = in[q] >= 0 ? at++ : leaf++;
#pragma unroll
        for (int k = 0; k < 4; ++k)   // a constant index keeps ref in registers
            if (k == to) ref[k] = in[q];
    }
}

// Heads (internal nodes at even depth) and the prefix sums of their
// internal-child counts: off[i] within the block of kHeadThreads numbers, the
// block's sum in sums; off is ~0 for the others.
__global__ void __launch_bounds__(kHeadThreads)
k_heads(const float4* __restrict__ nodes, const int32_t* __restrict__ parent, int n_inner, unsigned* __restrict__ off,
        unsigned* __restrict__ sums) {
    __shared__ unsigned warp_sum[kHeadThreads / 32];
    const int i = (int)blockIdx.x * kHeadThreads + (int)threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int root = n_inner - 1;
    bool head = false;
    int ni = 0;
    if (i < n_inner) {
        // a PLOC tree of 2^30 leaves can be deeper than a radix tree; the bound only
        // guards against a malformed parent array
        int d = 0;
        for (int q = root - i; q != root && d < 4096; ++d) q = parent[q];
        head = (d & 1) == 0;
        if (head) {
            int ref[4], m;
            children4(nodes, root - i, ref, m, ni);
        }
    }
    unsigned incl = (unsigned)ni;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    unsigned before = 0u, all = 0u;
#pragma unroll
    for (int w = 0; w < kHeadThreads / 32; ++w) {
        before += w < warp ? warp_sum[w] : 0u;
        all += warp_sum[w];
    }
    if (i < n_inner) off[i] = head ? before + incl - (unsigned)ni : 0xffffffffu;
    if (threadIdx.x == 0) sums[blockIdx.x] = all;
}

// Exclusive prefixes of nb sums in place, their total in *total; one block.
__global__ void __launch_bounds__(1024) k_scan_sums(unsigned* __restrict__ sums, int nb, unsigned* __restrict__ total) {
    __shared__ unsigned warp_sum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned carry = 0u;
    for (int base = 0; base < nb; base += 1024) {
        const int k = base + (int)threadIdx.x;
        const unsigned x = k < nb ? sums[k] : 0u;
        unsigned incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        unsigned before = 0u, all = 0u;
        for (int w = 0; w < 32; ++w) {
            const unsigned v = warp_sum[w];
            before += w < warp ? v : 0u;
            all += v;
        }
        if (k < nb) sums[k] = carry + before + incl - x;
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// Head of every 4-wide node: the root is node 0, the k-th internal child of
// head i node 1 + (internal children of the heads before i) + k.
__global__ void k_number4(const float4* __restrict__ nodes, const unsigned* __restrict__ off,
                          const unsigned* __restrict__ sums, int n_inner, int* __restrict__ head_of) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_inner) return;
    const unsigned o = off[i];
    if (o == 0xffffffffu) return;
    if (i == 0) head_of[0] = n_inner - 1;
    int ref[4], m, ni;
    children4(nodes, n_inner - 1 - i, ref, m, ni);
    const unsigned first = 1u + sums[i / kHeadThreads] + o;
    for (int k = 0; k < ni; ++k)
        if (first + (unsigned)k < (unsigned)n_inner) head_of[first + (unsigned)k] = ref[k];
}

// 4-wide node j from its head: six planes of the four child boxes, the child
// references (internal 4-wide indices, ~leaf, kEmptyRef for unused slots with
// a zero box) and the slot keys: kInner | q for an internal child in slot q, q
// for a leaf, all ones for an unused slot (the traversal sorts (entry distance |
// key) as integers).
// Four lanes to a node: lane q loads child q's box, and the four write the
// node's rows side by side, 64 bytes at a time (a thread writing all 256 bytes
// of a node took 63 us for the 343 K nodes of 1.07 M triangles, 41 us so).
__global__ void __launch_bounds__(kThreads)
k_pack_nodes4(const float4* __restrict__ nodes, const float* __restrict__ leaf_box, const unsigned* __restrict__ off,
              const unsigned* __restrict__ sums, const int* __restrict__ head_of, int n_inner, int n_nodes4,
              float4* __restrict__ nodes4) {
    const long long t = (long long)blockIdx.x * kThreads + threadIdx.x;
    const int j = (int)(t >> 2), q = (int)(t & 3);
    const int id = j < n_nodes4 ? head_of[j] : -1;
    const bool ok = (unsigned)id < (unsigned)n_inner;   // else past the end, or a malformed binary tree
    float b[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    int out = kEmptyRef;
    unsigned key = 0xffffffffu;
    if (ok) {
        const int i = n_inner - 1 - id;
        int ref[4], m, ni;
        children4(nodes, id, ref, m, ni);
        const int r = q == 0 ? ref[0] : (q == 1 ? ref[1] : (q == 2 ? ref[2] : ref[3]));
        if (q < ni) {
            out = (int)(1u + sums[i / kHeadThreads] + off[i]) + q;
            key = kInner | (unsigned)q;
        } else if (q < m) {
            out = r;
            key = (unsigned)q;
        }
        if (q < m && r >= 0) {
            const float4 l = nodes[2ll * r], h = nodes[2ll * r + 1];
            b[0] = l.x; b[1] = l.y; b[2] = l.z; b[3] = h.x; b[4] = h.y; b[5] = h.z;
        } else if (q < m) {
            const float* p = leaf_box + 6ll * ~r;
#pragma unroll
            for (int k = 0; k < 6; ++k) b[k] = p[k];
        }
    }
    float4* o = nodes4 + 16ll * j;
    const int lane0 = (int)(threadIdx.x & 31) & ~3;
    const bool lo_row = q == 0 || q == 3;   // per axis: lo, hi, hi, lo of the four children
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float l = __shfl_sync(0xffffffffu, b[a], lane0 + c), h = __shfl_sync(0xffffffffu, b[a + 3], lane0 + c);
            v[c] = lo_row ? l : h;
        }
        if (ok) o[4 * a + q] = make_float4(v[0], v[1], v[2], v[3]);
    }
    int v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int r = __shfl_sync(0xffffffffu, out, lane0 + c), k = __shfl_sync(0xffffffffu, (int)key, lane0 + c);
        v[c] = q == 0 ? r : (q == 1 ? k : 0);
    }
    if (ok) o[12 + q] = make_float4(__int_as_float(v[0]), __int_as_float(v[1]), __int_as_float(v[2]), __int_as_float(v[3]));
}

// The scratch block's arrays.  tree4_build leaves the binary tree, the heads'
// offsets and the heads of the 4-wide nodes for tree4_pack.
struct Tree4Scratch {
    float4 *clusters2, *nodes;
    int32_t* parent;
    unsigned char* fates;
    unsigned* counts;
    int2* scanned;
    PlocState* state;
    unsigned *off, *sums, *total;
    int* head_of;
    size_t bytes;
};

Tree4Scratch carve(void* scratch, int n) {
    char* p = static_cast<char*>(scratch);
    size_t at = 0;
    auto take = [&](auto** q, size_t count) {
        *q = reinterpret_cast<std::remove_reference_t<decltype(**q)>*>(p + at);
        at += (count * sizeof(**q) + 255) & ~(size_t)255;
    };
    const size_t N = (size_t)n;
    Tree4Scratch t;
    take(&t.clusters2, 2 * N);
    take(&t.nodes, 2 * N);
    take(&t.parent, N);
    take(&t.fates, N);
    take(&t.counts, N / kTile + 1);
    take(&t.scanned, N / kTile + 1);
    take(&t.state, 2);
    take(&t.off, N);
    take(&t.sums, N / kHeadThreads + 1);
    take(&t.total, 1);
    take(&t.head_of, N);
    t.bytes = at;
    return t;
}

}  // namespace

size_t tree4_scratch_bytes(int n) { return carve(nullptr, n > 1 ? n : 1).bytes; }

cudaError_t tree4_build(const LbvhBuffers& b, void* scratch, cudaStream_t s, int num_sms, int* n_nodes4) {
    const int n = b.n;
    *n_nodes4 = 0;
    if (n <= 1) return cudaSuccess;
    const int n_inner = n - 1;
    const Tree4Scratch sc = carve(scratch, n);
    Ploc p;
    p.clusters0 = b.clusters;
    p.clusters1 = sc.clusters2;
    p.nodes = sc.nodes;
    p.parent = sc.parent;
    p.fates = sc.fates;
    p.counts = sc.counts;
    p.state = sc.state;
    // the attribute is the current device's and context's: every build sets it
    const cudaError_t big = cudaFuncSetAttribute(k_ploc_tail, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)sizeof(TailShared));
    if (big != cudaSuccess) {
        cudaGetLastError();   // it is returned, not left for a later call
        return big;
    }
    k_ploc_start<<<1, 1, 0, s>>>(sc.state, n);
    count_launch(1);
    PlocState st{n, 0, 0, 0};
    int par = 0, rounds = 0;
    while (st.m > 1) {
        // the rounds that should bring the clusters to kTail at 82 % a round
        // (a few more: a round that finds kTail or fewer does nothing)
        int more = 0;
        if (st.m > kTail) more = 2 + (int)std::ceil(std::log((double)st.m / kTail) / std::log(1.0 / 0.83));
        if ((rounds += more) > kMaxRounds) return cudaErrorUnknown;
        const int blocks = blocks_for(st.m, kTile);
        int2* scanned = blocks > kScanBlocks ? sc.scanned : nullptr;
        double expected = blocks;
        for (int r = 0; r < more; ++r) {
            const unsigned grid = (unsigned)std::min(std::ceil(expected), 4.0 * num_sms);
            expected = std::max(1.0, 0.85 * expected);
            cudaError_t e = launch_overlapped(k_ploc_pair, grid, kRoundThreads, 0, s, p, par);
            if (e == cudaSuccess && scanned) e = launch_overlapped(k_ploc_scan, 1, 1024, 0, s, p, par, scanned);
            if (e == cudaSuccess) e = launch_overlapped(k_ploc_merge, grid, kRoundThreads, 0, s, p, par, scanned);
            if (e != cudaSuccess) return e;
            par ^= 1;
        }
        cudaError_t e = launch_overlapped(k_ploc_tail, 1, kTailThreads, sizeof(TailShared), s, p, par);
        PlocState now;
        if (e == cudaSuccess) e = cudaMemcpyAsync(&now, sc.state + par, sizeof(now), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
        if (now.stuck || now.m >= st.m) return cudaErrorUnknown;
        st = now;
    }
    if (st.nodes != n_inner) return cudaErrorUnknown;
    const int g = blocks_for(n_inner, kHeadThreads);
    k_heads<<<g, kHeadThreads, 0, s>>>(sc.nodes, sc.parent, n_inner, sc.off, sc.sums);
    k_scan_sums<<<1, 1024, 0, s>>>(sc.sums, g, sc.total);
    k_number4<<<blocks_for(n_inner, kThreads), kThreads, 0, s>>>(sc.nodes, sc.off, sc.sums, n_inner, sc.head_of);
    count_launch(3);
    cudaError_t e = cudaGetLastError();
    unsigned total = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&total, sc.total, sizeof(total), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the count is read next
    if (e != cudaSuccess) return e;
    const long long n4 = 1ll + total;   // the root and every head's internal children
    if (n4 > n_inner) return cudaErrorUnknown;
    *n_nodes4 = (int)n4;
    return cudaSuccess;
}

cudaError_t tree4_pack(const LbvhBuffers& b, void* scratch, int n_nodes4, cudaStream_t s) {
    const int n = b.n;
    if (n <= 1) return cudaSuccess;
    const Tree4Scratch sc = carve(scratch, n);
    k_pack_nodes4<<<blocks_for(4ll * n_nodes4, kThreads), kThreads, 0, s>>>(sc.nodes, b.leaf_box, sc.off, sc.sums,
                                                                            sc.head_of, n - 1, n_nodes4, b.nodes4);
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace vafr
