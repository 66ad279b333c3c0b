// lbvh.cu -- LBVH construction on the GPU (Karras 2012, "Maximizing Parallelism
// in the Construction of BVHs, Octrees, and k-d Trees"):
//   1. scene bounds of the triangle centroid sums s = (v0 + v1) + v2,
//   2. 30-bit Morton codes of s on a cubic grid of 1024 cells along the
//      largest extent of the bounds,
//   3. stable LSD radix sort of (code, triangle id), 4 passes of 8 bits,
//   4. sorted leaves: triangle box, 48-byte traversal leaf, the traversal
//      tree's first clusters,
//   5. binary radix tree: one thread per internal node,
//   6. bottom-up FP32 bounds, a node's second arrival writing its box and its
//      64-byte two-child traversal node.
// The quantisation uses explicitly rounded intrinsics (no FMA contraction) so
// the codes are bit-identical to any IEEE FP32 evaluation of the same sequence.
// No kernel here waits on another thread: there is nothing that can spin.
#include "vafr_internal.cuh"

#include <float.h>

#include <cuda.h>

#include <cstring>
#include <mutex>

namespace vafr {

size_t lbvh_sort_blocks(int n);

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kBoundsBlocks = 304;

__device__ __forceinline__ float centroid_sum(const float* t, int k) {
    return __fadd_rn(__fadd_rn(t[k], t[3 + k]), t[6 + k]);
}

__global__ void k_bounds_partial(const float* __restrict__ tris, int n, float* __restrict__ part) {
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float* t = tris + 9ll * i;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float s = centroid_sum(t, k);
            lo[k] = fminf(lo[k], s);
            hi[k] = fmaxf(hi[k], s);
        }
    }
    __shared__ float red[6][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
    }
    if (lane == 0) {
        for (int k = 0; k < 3; ++k) { red[k][warp] = lo[k]; red[3 + k][warp] = hi[k]; }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        float v = red[k][0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            v = k < 3 ? fminf(v, red[k][w]) : fmaxf(v, red[k][w]);
        part[6 * blockIdx.x + k] = v;
    }
}

// One warp per bound (a minimum or maximum over the blocks' partial bounds).
__global__ void k_bounds_final(const float* __restrict__ part, int nb, float* __restrict__ out) {
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float v = part[k];
    for (int b = lane; b < nb; b += 32) v = k < 3 ? fminf(v, part[6 * b + k]) : fmaxf(v, part[6 * b + k]);
    for (int o = 16; o > 0; o >>= 1) {
        const float w = __shfl_xor_sync(0xffffffffu, v, o);
        v = k < 3 ? fminf(v, w) : fmaxf(v, w);
    }
    if (lane == 0) out[k] = v;
}

// 10 bits spread to every third bit position (bit b -> bit 3b).
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
    x &= 0x3ffu;
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

__global__ void k_morton(const float* __restrict__ tris, int n, const float* __restrict__ bounds,
                         uint32_t* __restrict__ codes) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float* t = tris + 9ll * i;
    // cubic grid: every axis is scaled by the largest extent of the bounds
    const float ext = fmaxf(fmaxf(__fsub_rn(bounds[3], bounds[0]), __fsub_rn(bounds[4], bounds[1])),
                            __fsub_rn(bounds[5], bounds[2]));
    uint32_t q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float lo = bounds[k];
        if (!(ext > 0.0f)) { q[k] = 0u; continue; }
        const float s = centroid_sum(t, k);
        const float u = __fdiv_rn(__fsub_rn(s, lo), ext);
        const uint32_t c = __float2uint_rz(__fmul_rn(u, 1024.0f));
        q[k] = c > 1023u ? 1023u : c;
    }
    codes[i] = (spread3(q[0]) << 2) | (spread3(q[1]) << 1) | spread3(q[2]);
}

// ---- stable LSD radix sort ----------------------------------------------------
// Pass = histogram (per tile) -> exclusive scan in (digit, tile) order ->
// scatter.  The scatter ranks keys of a tile stably with warp multi-split:
// every warp owns a contiguous run of the tile and walks it 32 keys at a time
// in index order; __match_any_sync groups equal digits, and a per-(warp,
// digit) counter accumulates ranks; a prefix over warps then orders warps.

__global__ void k_radix_hist(const uint32_t* __restrict__ keys, int n, int shift,
                             unsigned* __restrict__ hist, int nblocks) {
    __shared__ unsigned h[256];
    h[threadIdx.x] = 0u;
    __syncthreads();
    const long long base = (long long)blockIdx.x * kSortTile;
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const long long i = base + it * kSortThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[(size_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Block d scans digit d's counters over the tiles (exclusive, in place) and
// leaves their sum in total[d]; the scatter adds the smaller digits' totals.
// A single block scanning all 256 x tiles counters took 110 us of each pass at
// 1.07 M keys (134 K counters); 256 blocks take 4 us.
__global__ void __launch_bounds__(kSortThreads) k_radix_rows(unsigned* __restrict__ hist, int nblocks,
                                                             unsigned* __restrict__ total) {
    __shared__ unsigned warp_sum[kSortWarps];
    unsigned* row = hist + (size_t)blockIdx.x * nblocks;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned carry = 0u;
    for (int base = 0; base < nblocks; base += kSortThreads) {
        const int i = base + (int)threadIdx.x;
        const unsigned x = i < nblocks ? row[i] : 0u;
        unsigned incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        unsigned before = 0u, all = 0u;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const unsigned c = warp_sum[w];
            before += w < warp ? c : 0u;
            all += c;
        }
        if (i < nblocks) row[i] = carry + before + incl - x;
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(kSortThreads)
k_radix_scatter(const uint32_t* __restrict__ kin, const int32_t* __restrict__ vin,
                uint32_t* __restrict__ kout, int32_t* __restrict__ vout, int n, int shift,
                const unsigned* __restrict__ hist, int nblocks, const unsigned* __restrict__ total) {
    __shared__ unsigned cnt[kSortWarps][256];
    __shared__ unsigned gbase[256];
    __shared__ unsigned warp_sum[kSortWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kSortWarps * 256; i += kSortThreads) (&cnt[0][0])[i] = 0u;
    {   // first slot of this tile's keys with digit threadIdx.x
        const unsigned x = total[threadIdx.x];
        unsigned incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        unsigned before = 0u;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) before += w < warp ? warp_sum[w] : 0u;
        gbase[threadIdx.x] = before + incl - x + hist[(size_t)threadIdx.x * nblocks + blockIdx.x];
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    const long long base = (long long)blockIdx.x * kSortTile + (long long)warp * (32 * kSortItems);
    uint32_t key[kSortItems];
    int32_t val[kSortItems];
    unsigned rank[kSortItems], dig[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const long long i = base + r * 32 + lane;
        const bool valid = i < n;
        key[r] = valid ? kin[i] : 0u;
        val[r] = valid ? (vin ? vin[i] : (int32_t)i) : 0;
        const unsigned d = valid ? ((key[r] >> shift) & 255u) : 256u + lane;
        dig[r] = d;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        unsigned before = 0u;
        if (valid) before = cnt[warp][d];
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) cnt[warp][d] = before + __popc(peers);
        __syncwarp();
        rank[r] = before + __popc(peers & lt);
    }
    __syncthreads();
    {
        const int d = threadIdx.x;   // kSortThreads == 256 digits
        unsigned run = 0u;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const unsigned c = cnt[w][d];
            cnt[w][d] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const long long i = base + r * 32 + lane;
        if (i < n) {
            const unsigned d = dig[r];
            const unsigned dst = gbase[d] + cnt[warp][d] + rank[r];
            kout[dst] = key[r];
            vout[dst] = val[r];
        }
    }
}

// ---- Karras hierarchy -----------------------------------------------------------
// delta(i, j): common prefix length of the keys (code, index); -1 out of range.
__device__ __forceinline__ int delta(const uint32_t* __restrict__ k, int n, int i, int j, uint32_t ki) {
    if (j < 0 || j >= n) return -1;
    const uint32_t kj = k[j];
    if (kj == ki) return 32 + __clz((unsigned)(i ^ j));
    return __clz(ki ^ kj);
}

// links[i] = (left, right, other end of node i's leaves, parent): what a climb
// needs of a node in one load.  A node's thread writes all but the parent,
// which its parent's thread writes.
__global__ void k_karras(const uint32_t* __restrict__ keys, int n, int2* __restrict__ child,
                         int4* __restrict__ links, int32_t* __restrict__ leaf_parent) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    const uint32_t ki = keys[i];
    const int d = (delta(keys, n, i, i + 1, ki) - delta(keys, n, i, i - 1, ki)) >= 0 ? 1 : -1;
    const int dmin = delta(keys, n, i, i - d, ki);
    int lmax = 2;
    while (delta(keys, n, i, i + lmax * d, ki) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(keys, n, i, i + (l + t) * d, ki) > dmin) l += t;
    const int j = i + l * d;
    const int dnode = delta(keys, n, i, j, ki);
    int s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (delta(keys, n, i, i + (s + t) * d, ki) > dnode) s += t;
    } while (t > 1);
    const int gamma = i + s * d + min(d, 0);
    const int lo = min(i, j), hi = max(i, j);
    const int L = (lo == gamma) ? ~gamma : gamma;
    const int R = (hi == gamma + 1) ? ~(gamma + 1) : gamma + 1;
    child[i] = make_int2(L, R);
    *reinterpret_cast<int2*>(&links[i]) = make_int2(L, R);
    links[i].z = j;
    *(L >= 0 ? &links[L].w : &leaf_parent[~L]) = i;
    *(R >= 0 ? &links[R].w : &leaf_parent[~R]) = i;
    if (i == 0) links[0].w = -1;
}

__device__ __forceinline__ void load_box(const float* p, float b[6]) {
#pragma unroll
    for (int k = 0; k < 6; ++k) b[k] = __ldcg(p + k);
}

__device__ __forceinline__ void merge_box(float b[6], const float a[6]) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        b[q] = fminf(b[q], a[q]);
        b[3 + q] = fmaxf(b[3 + q], a[3 + q]);
    }
}

// Bottom-up bounds: a thread per leaf climbs; at every internal node the first
// arrival stops and the second, which then has both children's boxes, writes
// the node's box and its two-child traversal node and continues.
// In k_refit_block a block takes kRefitLeaves consecutive leaves and makes the
// nodes whose leaves all lie among them: the children meet in shared memory.
// The few nodes above, one in some hundred, are left to k_refit_top, which
// climbs on from the listed children; there each arrival costs a device-wide
// fence and an atomic.  (One kernel for both kept a block's place on its SM
// for as long as its last thread climbed to the top: 143 us at 1.07 M leaves;
// every node in global memory and the traversal nodes packed in a pass of
// their own 176 us; the two kernels 69 + 52 us.)
constexpr int kRefitLeaves = 512;

// A child whose parent is the next to be made: box b, its sibling's box a.
__device__ __forceinline__ void make_parent(int node, int2 kids, int side, float b[6], const float a[6],
                                            float* __restrict__ node_box, float4* __restrict__ nodes) {
    float L[6], R[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        L[q] = side ? a[q] : b[q];
        R[q] = side ? b[q] : a[q];
    }
    // per axis: (left lo, right lo, left hi, right hi), so both children's
    // slabs are computed with paired FP32 instructions
    float4* nd = nodes + 4ll * node;
#pragma unroll
    for (int q = 0; q < 3; ++q) nd[q] = make_float4(L[q], R[q], L[q + 3], R[q + 3]);
    nd[3] = make_float4(__int_as_float(kids.x), __int_as_float(kids.y), 0.0f, 0.0f);
    merge_box(b, a);
    float* o = node_box + 6ll * node;
#pragma unroll
    for (int q = 0; q < 6; ++q) __stcg(o + q, b[q]);
}

__global__ void __launch_bounds__(kRefitLeaves)
k_refit_block(int n, const int4* __restrict__ links, const int32_t* __restrict__ leaf_parent,
              float* __restrict__ node_box, const float* __restrict__ leaf_box, float4* __restrict__ nodes,
              int* __restrict__ list, unsigned* __restrict__ listed) {
    __shared__ unsigned met[kRefitLeaves];
    __shared__ float box[2][6][kRefitLeaves];   // [child side][bound][node - b0]
    __shared__ int4 link[kRefitLeaves];
    __shared__ int up[kRefitLeaves];            // children whose parent has other leaves too
    __shared__ unsigned ups, at;
    const int b0 = (int)blockIdx.x * kRefitLeaves;
    const int k = b0 + (int)threadIdx.x;
    met[threadIdx.x] = 0u;
    if (threadIdx.x == 0) ups = 0u;
    if (k < n - 1) link[threadIdx.x] = links[k];
    __syncthreads();
    if (k < n) {
        float b[6];
        load_box(leaf_box + 6ll * k, b);
        int ref = ~k;
        int node = leaf_parent[k];
        while (node >= 0) {
            const int s = node - b0;   // a node's index is one end of its leaves
            if ((unsigned)s >= (unsigned)kRefitLeaves || (unsigned)(link[s].z - b0) >= (unsigned)kRefitLeaves) {
                const unsigned q = atomicAdd(&ups, 1u);   // a leaf's thread gets here at most once
                up[q] = ref;
                break;
            }
            const int2 c = make_int2(link[s].x, link[s].y);
            const int side = c.x == ref ? 0 : 1;
#pragma unroll
            for (int q = 0; q < 6; ++q) box[side][q][s] = b[q];
            __threadfence_block();
            if (atomicAdd(&met[s], 1u) != 1u) break;   // the first arrival; anything else only in a malformed tree
            __threadfence_block();
            float a[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) a[q] = *(volatile float*)&box[side ^ 1][q][s];
            make_parent(node, c, side, b, a, node_box, nodes);
            ref = node;
            node = link[s].w;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) at = ups ? atomicAdd(listed, ups) : 0u;
    __syncthreads();
    if (threadIdx.x < ups) list[at + threadIdx.x] = up[threadIdx.x];
}

__global__ void __launch_bounds__(256)
k_refit_top(int n, const int4* __restrict__ links, const int32_t* __restrict__ leaf_parent,
            unsigned* __restrict__ flags, float* __restrict__ node_box, const float* __restrict__ leaf_box,
            float4* __restrict__ nodes, const int* __restrict__ list, const unsigned* __restrict__ listed) {
    const unsigned count = min(*listed, (unsigned)n);
    for (unsigned q = blockIdx.x * 256 + threadIdx.x; q < count; q += gridDim.x * 256) {
        int ref = list[q];
        float b[6];
        load_box(ref >= 0 ? node_box + 6ll * ref : leaf_box + 6ll * ~ref, b);
        int node = ref >= 0 ? links[ref].w : leaf_parent[~ref];
        // a binary radix tree over 30-bit codes + 32-bit positions is at most 64
        // levels deep; the bound only guards against a malformed parent array
        int4 next = node >= 0 ? links[node] : make_int4(0, 0, 0, -1);
        for (int climb = 0; node >= 0 && climb < 96; ++climb) {
            const int4 ln = next;
            if (ln.w >= 0) next = links[ln.w];   // on its way while the arrival is counted
            __threadfence();   // this child's box, if written here, before its arrival
            if (atomicAdd(&flags[node], 1u) == 0u) break;
            __threadfence();
            const int2 c = make_int2(ln.x, ln.y);
            const int side = c.x == ref ? 0 : 1;
            const int sib = side ? c.x : c.y;
            float a[6];
            load_box(sib >= 0 ? node_box + 6ll * sib : leaf_box + 6ll * ~sib, a);
            make_parent(node, c, side, b, a, node_box, nodes);
            ref = node;
            node = ln.w;
        }
    }
}

__device__ __forceinline__ bool lex_less(float ax, float ay, float az, float bx, float by, float bz) {
    return ax < bx || (ax == bx && (ay < by || (ay == by && az < bz)));
}

// Sorted leaf k: its triangle's box, its traversal leaf, and the cluster that
// the traversal tree starts from (box with the reference ~k in lo.w).
// Leaves store their vertices in lexicographic (x, y, z) order.  The
// intersection test is two-sided, so the order carries no meaning, and
// identical triangles given with different vertex orders then evaluate to
// bit-identical t: the lower-id rule, not rounding, decides between them.
__global__ void k_leaves(const float* __restrict__ tris, const float* __restrict__ albedo,
                         const int32_t* __restrict__ ids, int n, float* __restrict__ leaf_box,
                         float4* __restrict__ leaves, float4* __restrict__ clusters,
                         float4* __restrict__ albedo4) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int id = ids[k];
    const float* t = tris + 9ll * id;
    float v[3][3], lo[3], hi[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) v[a][c] = t[3 * a + c];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lo[c] = fminf(fminf(v[0][c], v[1][c]), v[2][c]);
        hi[c] = fmaxf(fmaxf(v[0][c], v[1][c]), v[2][c]);
        leaf_box[6ll * k + c] = lo[c];
        leaf_box[6ll * k + 3 + c] = hi[c];
    }
    clusters[2ll * k] = make_float4(lo[0], lo[1], lo[2], __int_as_float(~k));
    clusters[2ll * k + 1] = make_float4(hi[0], hi[1], hi[2], 0.0f);
    // three-element sorting network
#define VAFR_CSWAP(i, j)                                                                      \
    if (lex_less(v[j][0], v[j][1], v[j][2], v[i][0], v[i][1], v[i][2])) {                     \
        for (int c = 0; c < 3; ++c) { const float q = v[i][c]; v[i][c] = v[j][c]; v[j][c] = q; } \
    }
    VAFR_CSWAP(0, 1)
    VAFR_CSWAP(1, 2)
    VAFR_CSWAP(0, 1)
#undef VAFR_CSWAP
    leaves[3ll * k + 0] = make_float4(v[0][0], v[0][1], v[0][2], __int_as_float(id));
    leaves[3ll * k + 1] = make_float4(v[1][0], v[1][1], v[1][2], 0.0f);
    leaves[3ll * k + 2] = make_float4(v[2][0], v[2][1], v[2][2], 0.0f);
    // albedo in original order (thread k writes triangle k's albedo)
    if (albedo)
        albedo4[k] = make_float4(albedo[3ll * k], albedo[3ll * k + 1], albedo[3ll * k + 2], 0.0f);
    else
        albedo4[k] = make_float4(0.8f, 0.8f, 0.8f, 0.0f);
}

inline int blocks_for(long long n, int tpb) { return (int)((n + tpb - 1) / tpb); }

// Morton codes of the triangles, then the stable (code, id) order: codes in
// input order stay in `codes`, the sorted keys and ids end in `keys` and `ids`.
// `hist` holds 256 counters per tile and 256 totals.
void morton_sort(const float* tris, int n, float* part_bounds, float* scene_bounds, uint32_t* codes,
                 uint32_t* keys_tmp, int32_t* ids_tmp, uint32_t* keys, int32_t* ids, unsigned* hist, cudaStream_t s) {
    const int nb_bounds = min(kBoundsBlocks, blocks_for(n, 256));
    k_bounds_partial<<<nb_bounds, 256, 0, s>>>(tris, n, part_bounds);
    k_bounds_final<<<1, 192, 0, s>>>(part_bounds, nb_bounds, scene_bounds);
    k_morton<<<blocks_for(n, 256), 256, 0, s>>>(tris, n, scene_bounds, codes);
    count_launch(3);
    const int nblocks = (int)lbvh_sort_blocks(n);
    unsigned* total = hist + 256ull * nblocks;
    // ping-pong: codes -> tmp -> sorted -> tmp -> sorted
    const uint32_t* kin = codes;
    const int32_t* vin = nullptr;
    for (int pass = 0; pass < 4; ++pass) {
        uint32_t* kout = (pass & 1) ? keys : keys_tmp;
        int32_t* vout = (pass & 1) ? ids : ids_tmp;
        k_radix_hist<<<nblocks, kSortThreads, 0, s>>>(kin, n, 8 * pass, hist, nblocks);
        k_radix_rows<<<256, kSortThreads, 0, s>>>(hist, nblocks, total);
        k_radix_scatter<<<nblocks, kSortThreads, 0, s>>>(kin, vin, kout, vout, n, 8 * pass, hist, nblocks, total);
        count_launch(3);
        kin = kout;
        vin = vout;
    }
}

}  // namespace

size_t lbvh_sort_blocks(int n) { return (size_t)((n + kSortTile - 1) / kSortTile); }
size_t lbvh_hist_elems(int n) { return 256 * (lbvh_sort_blocks(n) + 1); }

cudaError_t lbvh_sort(const LbvhBuffers& b, cudaStream_t s) {
    const int n = b.n;
    if (n <= 0) return cudaSuccess;
    morton_sort(b.tris, n, b.part_bounds, b.scene_bounds, b.codes, b.keys_tmp, b.ids_tmp, b.keys_sorted, b.ids,
                b.hist, s);
    k_leaves<<<blocks_for(n, 256), 256, 0, s>>>(b.tris, b.albedo, b.ids, n, b.leaf_box, b.leaves, b.clusters,
                                                b.albedo4);
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t lbvh_hierarchy(const LbvhBuffers& b, cudaStream_t s) {
    const int n = b.n;
    if (n <= 1) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(b.flags, 0, sizeof(unsigned) * (size_t)n, s);   // n - 1 nodes, the list's length
    if (e != cudaSuccess) return e;
    unsigned* listed = b.flags + (n - 1);
    k_karras<<<blocks_for(n - 1, 256), 256, 0, s>>>(b.keys_sorted, n, b.child, b.links, b.leaf_parent);
    k_refit_block<<<blocks_for(n, kRefitLeaves), kRefitLeaves, 0, s>>>(n, b.links, b.leaf_parent, b.node_box,
                                                                       b.leaf_box, b.nodes, b.climbers, listed);
    k_refit_top<<<min(blocks_for(n, 256), 304), 256, 0, s>>>(n, b.links, b.leaf_parent, b.flags, b.node_box, b.leaf_box,
                                                             b.nodes, b.climbers, listed);
    count_launch(3);
    return cudaGetLastError();
}

}  // namespace vafr

// ---- allocation-free Morton codes + sort ---------------------------------------
// vafr_morton_sort_noalloc serves callers that may not allocate device memory:
// code running where the whole GPU's memory belongs to the caller's own pool
// allocator, or on a latency-critical thread where cudaMalloc's implicit
// device synchronisation is not acceptable.  All of its scratch lives in one
// file-scope __device__ array; it launches the same kernels as the build.
namespace vafr {
namespace {

constexpr int kNoAllocMaxTris = VAFR_NOALLOC_MAX_TRIS;
constexpr int kNoAllocBlocks = (kNoAllocMaxTris + kSortTile - 1) / kSortTile;

struct NoAllocScratch {
    uint32_t keys_tmp[kNoAllocMaxTris];
    int32_t ids_tmp[kNoAllocMaxTris];
    uint32_t keys_sorted[kNoAllocMaxTris];
    unsigned hist[256 * (kNoAllocBlocks + 1)];
    float part_bounds[6 * kBoundsBlocks];
    float scene_bounds[8];
};

// Held by every GPU that loads the library until the process exits
// (sizeof(NoAllocScratch) = 6.3 MB).  Every call shares it; nothing in it has
// to start at zero (each pass overwrites what it reads).
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
struct NoAllocSlot {
    NoAllocScratch* ptr;         // device address of the array, or nullptr
    unsigned long long ctx_id;   // context it was looked up in (0: unknown)
};
NoAllocSlot g_noalloc_slot[kNoAllocMaxDevices] = {};

// Process-unique id of the calling thread's current context, or 0 if the
// driver cannot say.  A device reset destroys the context and the module with
// the array; the context that replaces it has a new id, which tells the cache
// below to look the address up again.  The two driver calls are found
// through the runtime, so the library needs no link against the driver.
unsigned long long current_context_id() {
    using GetCur = CUresult (*)(CUcontext*);
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    static GetCur get_cur = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            get_cur = reinterpret_cast<GetCur>(f);
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
    });
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (!get_cur || !get_id || get_cur(&c) != CUDA_SUCCESS || !c || get_id(c, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// Device address of the scratch array on the current device.  In host code the
// array's name is only a host-side stand-in, so the address is looked up with
// that device current: once per device, and again after a device reset.
cudaError_t noalloc_scratch(NoAllocScratch** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
    const unsigned long long ctx = current_context_id();
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoAllocSlot& slot = g_noalloc_slot[dev];
    if (!slot.ptr || slot.ctx_id != ctx) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        slot = NoAllocSlot{static_cast<NoAllocScratch*>(p), ctx};
    }
    *out = slot.ptr;
    return cudaSuccess;
}

// Whether byte ranges [a, a + na) and [b, b + nb) share a byte.
bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
}

}  // namespace
}  // namespace vafr

extern "C" VAFR_API int vafr_morton_sort_noalloc(const float* tri_xyz, int64_t n_tris,
                                                 uint32_t* codes_out, int32_t* sorted_ids_out,
                                                 void* stream, char* err, int32_t err_len) {
    using namespace vafr;
    auto report = [&](int code, const char* msg) {
        if (err && err_len > 0) {
            std::strncpy(err, msg, (size_t)err_len - 1);
            err[err_len - 1] = '\0';
        }
        return code;
    };
    if (n_tris < 0) return report(VAFR_ERR_INVALID_ARG, "n_tris is negative");
    if (n_tris > kNoAllocMaxTris)
        return report(VAFR_ERR_INVALID_ARG, "n_tris exceeds VAFR_NOALLOC_MAX_TRIS (524288)");
    if (n_tris == 0) return VAFR_OK;
    if (!tri_xyz || !codes_out || !sorted_ids_out) return report(VAFR_ERR_INVALID_ARG, "NULL pointer");
    for (const void* p : {(const void*)tri_xyz, (const void*)codes_out, (const void*)sorted_ids_out}) {
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, p) != cudaSuccess ||
            (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)) {
            cudaGetLastError();
            return report(VAFR_ERR_INVALID_ARG, "every buffer must be device memory");
        }
    }
    // the sort reads its input keys while writing the output ids: any shared
    // byte between the three buffers would corrupt the result silently
    const size_t nt = (size_t)n_tris;
    if (overlaps(codes_out, 4 * nt, sorted_ids_out, 4 * nt) || overlaps(tri_xyz, 36 * nt, codes_out, 4 * nt) ||
        overlaps(tri_xyz, 36 * nt, sorted_ids_out, 4 * nt))
        return report(VAFR_ERR_INVALID_ARG, "tri_xyz, codes_out and sorted_ids_out must not overlap");
    NoAllocScratch* sc = nullptr;
    cudaError_t e = noalloc_scratch(&sc);
    if (e != cudaSuccess) return report(VAFR_ERR_CUDA, cudaGetErrorString(e));
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int n = (int)n_tris;
    morton_sort(tri_xyz, n, sc->part_bounds, sc->scene_bounds, codes_out, sc->keys_tmp, sc->ids_tmp, sc->keys_sorted,
                sorted_ids_out, sc->hist, s);
    e = cudaGetLastError();
    if (e != cudaSuccess) return report(VAFR_ERR_CUDA, cudaGetErrorString(e));
    return VAFR_OK;
}
