// fxaa.cu -- anti-aliasing inside the LP buffer (Sec. 3.4: the LP buffer gets
// FXAA before the inverse mapping; Sec. 7 ablates it).  The paper names FXAA
// (Lottes 2009) without parameters; this is that method on the LP grid:
//
//   grid    texel (c, j); along the angle its neighbours are rows j -+ 1 of
//           column c (the guard slots hold the wrap); across the radius,
//           column c' = c -+ 1 (clamped to [0, C-1]) contributes its texel
//           whose angular interval holds the angle of (c, j):
//           j' = floor((2j + 1) n_c' / (2 n_c)).
//   luma    0.299 R + 0.587 G + 0.114 B.
//   1 skip    luma range of {M, N, S, E, W} below max(1/12, max/6): copy.
//   2 axis    second differences across the angle (kA) and across the radius
//             (kR) over the 3 x 3 neighbourhood; kR >= kA: the blend steps a
//             column and the edge is walked along the angle, else the reverse.
//   3 side    blend towards the neighbour with the larger luma step (the
//             positive one on a tie); mid-line luma = their mean, threshold
//             a quarter of the step.
//   4 search  up to 12 unit steps each way along the edge; a step averages
//             the luma of the walked texel and of its partner across the
//             edge; the end is where that leaves the mid-line by the threshold.
//   5 offset  1/2 - d/D from the nearer end (d) and both ends (D), when that
//             end's luma lies across the mid-line from the texel's.
//   6 subpix  a = |3x3 mean (edges 2, corners 1) - M| / range;
//             ((3 - 2a) a^2)^2 x 3/4.
//   7 blend   texel + max(offset, subpix) (neighbour - texel), every channel.
// Luma and every branch decision use FP32 in one fixed order (no contraction),
// offsets and the blend FP32.  Two passes: the luma of every slot into a scratch
// array, then, in the frame's screen-space Hilbert order, the filter, which
// reads lumas (4 bytes) for its neighbourhood and search and colours only for
// the texel and its blend partner.  The output (a second LP buffer) gets the
// guard copies too.
#include "vafr_internal.cuh"

namespace vafr {
namespace {

constexpr int kFxaaSteps = 12;

__device__ __forceinline__ float4 ld_texel(const void* lp, int fmt, int slot) {
    if (fmt == VAFR_FMT_RGBA16F) {
        const uint2 p = reinterpret_cast<const uint2*>(lp)[slot];
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&p.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&p.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return reinterpret_cast<const float4*>(lp)[slot];
}

__device__ __forceinline__ void st_texel(void* lp, int fmt, int slot, float4 v) {
    if (fmt == VAFR_FMT_RGBA16F) {
        const __half2 lo = __floats2half2_rn(v.x, v.y), hi = __floats2half2_rn(v.z, v.w);
        uint2 p;
        p.x = *reinterpret_cast<const unsigned*>(&lo);
        p.y = *reinterpret_cast<const unsigned*>(&hi);
        reinterpret_cast<uint2*>(lp)[slot] = p;
    } else {
        reinterpret_cast<float4*>(lp)[slot] = v;
    }
}

__device__ __forceinline__ float luma_of(float4 c) {
    float y = __fmul_rn(0.299f, c.x);
    y = __fadd_rn(y, __fmul_rn(0.587f, c.y));
    return __fadd_rn(y, __fmul_rn(0.114f, c.z));
}

// floor(num / D) for a divisor D = 2 n_c fixed per texel: with num < 2^24 the
// FP32 product num * (1/D) is within one of the quotient (relative error
// <= 2^-23 and quotients < 2^16), fixed by one step each way; larger
// numerators divide in integers.
struct RowDiv {
    unsigned D;
    float rD;
    __device__ __forceinline__ explicit RowDiv(int n) : D(2u * (unsigned)n), rD(1.0f / (float)(2 * n)) {}
    __device__ __forceinline__ int operator()(unsigned num) const {
        if (num >= (1u << 24)) return (int)(num / D);
        unsigned q = (unsigned)((float)num * rD);
        q += (q + 1u) * D <= num ? 1u : 0u;
        q -= q * D > num ? 1u : 0u;
        return (int)q;
    }
};

struct Grid {
    const int2* col;   // (slot of row 0, count)
    int C;
    const void* lp;
    int fmt;
    const float* lum;  // luma of every slot (guards included)

    // slot of the texel of column c2 (clamped) at the angle of row j of column
    // c, moved dj rows; |dj| <= 1 may land on a guard slot.  The row is
    // floor((2j + 1) n_c2 / (2 n_c)): the one whose angular interval holds the
    // centre of row j.
    __device__ __forceinline__ int at(int c, int j, const RowDiv& div, int c2, int dj) const {
        c2 = min(max(c2, 0), C - 1);
        const int2 cc = __ldg(col + c2);
        const unsigned long long num = (unsigned long long)(2 * j + 1) * (unsigned)cc.y;
        const int j2 = c2 == c ? j
                               : (num < (1ull << 32) ? div((unsigned)num) : (int)(num / div.D));
        return cc.x + j2 + dj;
    }
    __device__ __forceinline__ float luma(int slot) const { return lum[slot]; }
};

__device__ __forceinline__ float abs_second_diff(float a, float b, float m) {
    return fabsf(__fsub_rn(__fadd_rn(a, b), __fmul_rn(2.0f, m)));
}

// A texel (c, j) (slot t, count n) with its luma and its neighbours'; the
// radial neighbours' angular neighbours are the slots beside them.
struct Cross {
    int sE, sW;
    float M, N, S, E, W, range, hi;
    __device__ __forceinline__ Cross(const Grid& g, int c, int j, const RowDiv& div, int t) {
        sE = g.at(c, j, div, c + 1, 0);
        sW = g.at(c, j, div, c - 1, 0);
        M = g.luma(t);
        N = g.luma(t + 1);
        S = g.luma(t - 1);
        E = g.luma(sE);
        W = g.luma(sW);
        const float lo = fminf(M, fminf(fminf(N, S), fminf(E, W)));
        hi = fmaxf(M, fmaxf(fmaxf(N, S), fmaxf(E, W)));
        range = __fsub_rn(hi, lo);
    }
    // step 1: no edge here
    __device__ __forceinline__ bool flat() const {
        return range < fmaxf(1.0f / 12.0f, __fmul_rn(hi, 1.0f / 6.0f));
    }
};

// The filtered colour of an edge texel (c, j) (slot t, count n).
__device__ __forceinline__ float4 fxaa_edge(const Grid& g, int c, int j, int n, int t) {
    const RowDiv div(n);
    const Cross x(g, c, j, div, t);
    const int sE = x.sE, sW = x.sW;
    const float M = x.M, N = x.N, S = x.S, E = x.E, W = x.W, range = x.range;
    const float4 cM = ld_texel(g.lp, g.fmt, t);
    const float NE = g.luma(sE + 1), SE = g.luma(sE - 1);
    const float NW = g.luma(sW + 1), SW = g.luma(sW - 1);
    // 2 axis
    const float kA = __fadd_rn(__fadd_rn(__fmul_rn(2.0f, abs_second_diff(N, S, M)), abs_second_diff(NE, SE, E)),
                               abs_second_diff(NW, SW, W));
    const float kR = __fadd_rn(__fadd_rn(__fmul_rn(2.0f, abs_second_diff(E, W, M)), abs_second_diff(NE, NW, N)),
                               abs_second_diff(SE, SW, S));
    const bool across_cols = kR >= kA;
    // 3 side
    const float Ln = across_cols ? W : S, Lp = across_cols ? E : N;
    const float gn = fabsf(__fsub_rn(Ln, M)), gp = fabsf(__fsub_rn(Lp, M));
    const bool pos = gp >= gn;
    const float avg = __fmul_rn(0.5f, __fadd_rn(M, pos ? Lp : Ln));
    const float thr = __fmul_rn(0.25f, fmaxf(gn, gp));
    const int side = pos ? 1 : -1;
    const int2 cc = __ldg(g.col + c);
    // 4 search
    int dist[2];
    float end[2];
    // along the rows of column c, the partner column's row at the walked texel's
    // angle is a quotient whose numerator steps by 2 n_partner: it is kept with
    // its remainder instead of divided for at every step
    const int cp = min(max(c + side, 0), g.C - 1);
    const int2 pc = __ldg(g.col + cp);
    const long long num0 = (long long)(2 * j + 1) * pc.y;
    const int q0 = cp == c ? j : (pos ? sE : sW) - pc.x;
    const int rem0 = (int)(num0 - (long long)q0 * (2 * n));   // in [0, 2n)
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        const int sgn = d ? 1 : -1;
        dist[d] = kFxaaSteps;
        end[d] = 0.0f;
        int jk = j, q = q0, rem = rem0;
#pragma unroll 1
        for (int k = 1; k <= kFxaaSteps; ++k) {
            int ta, tb;
            if (across_cols) {   // walk the rows of column c
                jk += sgn;
                rem += sgn * 2 * pc.y;
                if (jk < 0 || jk == n) {   // the wrap: all of the partner's rows fewer or more
                    jk -= sgn * n;
                    q -= sgn * pc.y;
                }
                while (rem < 0) { rem += 2 * n; --q; }
                while (rem >= 2 * n) { rem -= 2 * n; ++q; }
                ta = cc.x + jk;
                tb = cp == c ? ta : pc.x + q;
            } else {             // walk the columns at the angle of (c, j)
                ta = g.at(c, j, div, c + sgn * k, 0);
                tb = ta + side;
            }
            const float s = __fmul_rn(0.5f, __fadd_rn(g.luma(ta), g.luma(tb)));
            end[d] = s;
            if (fabsf(__fsub_rn(s, avg)) >= thr) {
                dist[d] = k;
                break;
            }
        }
    }
    // 5 offset
    const bool near_neg = dist[0] < dist[1];
    const int dn = near_neg ? dist[0] : dist[1];
    const float lend = near_neg ? end[0] : end[1];
    const bool good = (__fsub_rn(lend, avg) < 0.0f) != (__fsub_rn(M, avg) < 0.0f);
    const float off_edge = good ? 0.5f - (float)dn / (float)(dist[0] + dist[1]) : 0.0f;
    // 6 subpix
    const float l3 = (2.0f * (N + S + E + W) + (NE + NW + SE + SW)) * (1.0f / 12.0f);
    const float a = fminf(fabsf(l3 - M) / range, 1.0f);
    const float bsub = (3.0f - 2.0f * a) * a * a;
    const float w = fmaxf(off_edge, bsub * bsub * 0.75f);
    // 7 blend
    const float4 q = ld_texel(g.lp, g.fmt, across_cols ? (pos ? sE : sW) : t + side);
    return make_float4(fmaf(w, q.x - cM.x, cM.x), fmaf(w, q.y - cM.y, cM.y), fmaf(w, q.z - cM.z, cM.z),
                       fmaf(w, q.w - cM.w, cM.w));
}

template <class B>
__device__ __forceinline__ int find_aa_frame(const B& b, long long w) {
    int lo = 0, hi = b.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (b.d[mid].aa_begin <= w) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Pass 1: the luma of every slot into the frame's scratch.  A block takes rows of
// one column (blockIdx.x; frame blockIdx.z), kLumaItems to a thread and all of them
// loaded before the first is stored; the guard slots get the lumas of the texels
// that they stand for, whatever the buffer's own guards hold.  It reads 17 MB and
// writes 4 for an eye in FP32, so what counts is loads in flight and blocks of about
// the same length (rings have up to some 1,640 rows): both passes take 33.9 us over
// buffers in turn with 128 threads of 7 rows, 34.4 with 8, 34.7 with 6 or 5, 34.0 with
// 256 threads of 7, 34.4 of 3, 35.3 with 64 of 7; a pass over the slots in order,
// which cannot tell a guard from a texel, 33.9.
constexpr int kLumaThreads = 128, kLumaItems = 7, kLumaParts = 2;

template <class B>
__global__ void __launch_bounds__(kLumaThreads) k_lp_luma(const __grid_constant__ B b) {
    const FrameDesc& f = b.d[blockIdx.z];
    if (!f.lp_aa || (int)blockIdx.x >= f.n_cols) return;
    const int2 cc = __ldg(f.col + blockIdx.x);   // the layout's, which no launch writes
    const int n = cc.y;
    after_previous();
    for (int j0 = (int)blockIdx.y * (kLumaThreads * kLumaItems) + (int)threadIdx.x; j0 < n;
         j0 += kLumaParts * kLumaThreads * kLumaItems) {
        float4 v[kLumaItems];
#pragma unroll
        for (int k = 0; k < kLumaItems; ++k)
            if (j0 + k * kLumaThreads < n) v[k] = ld_texel(f.lp, f.lp_fmt, cc.x + j0 + k * kLumaThreads);
#pragma unroll
        for (int k = 0; k < kLumaItems; ++k) {
            const int j = j0 + k * kLumaThreads;
            if (j >= n) break;
            const float y = luma_of(v[k]);
            f.luma[cc.x + j] = y;
            if (j == 0) f.luma[cc.x + n] = y;
            if (j == n - 1) f.luma[cc.x - 1] = y;
        }
    }
}

// A texel of the batch, and its filtered colour's place (guards included).
struct AaTexel {
    const FrameDesc* f;
    int c, j, n, t;
    template <class B>
    __device__ __forceinline__ AaTexel(const B& b, long long w) {
        f = &b.d[find_aa_frame(b, w)];
        const int2 tc = __ldg(f->work + (w - f->aa_begin));   // (slot, column)
        const int2 cc = __ldg(f->col + tc.y);
        c = tc.y;
        j = tc.x - cc.x;
        n = cc.y;
        t = tc.x;
    }
    __device__ __forceinline__ Grid grid() const { return Grid{f->col, f->n_cols, f->lp, f->lp_fmt, f->luma}; }
    __device__ __forceinline__ void store(float4 v) const {
        st_texel(f->lp_aa, f->lp_fmt, t, v);
        if (j == 0) st_texel(f->lp_aa, f->lp_fmt, t + n, v);       // guard after the column
        if (j == n - 1) st_texel(f->lp_aa, f->lp_fmt, t - n, v);   // guard before it
    }
};

// Pass 2: the filter.  A block takes as many texels as it has threads, copies
// the flat ones and lists the edges, which its first threads then filter side
// by side.  An LP buffer in FP32 takes 37 us, both passes, and 33.5 since their
// launches overlap (47 with 256 threads,
// each filtering its own texel, a quotient at every step of the search and the
// lumas in the work order; 40 without the list).  Larger blocks or several
// texels to a thread lose to the densest blocks, whose searches end the launch.
constexpr int kFilterThreads = 128;

template <class B>
__global__ void __launch_bounds__(kFilterThreads, 10) k_fxaa_lp(const __grid_constant__ B b) {
    __shared__ unsigned short edges[kFilterThreads];
    __shared__ int n_edges;
    if (threadIdx.x == 0) n_edges = 0;
    after_previous();
    __syncthreads();
    const long long w0 = (long long)blockIdx.x * kFilterThreads;
    const int lane = threadIdx.x & 31;
    bool edge = false;
    if (w0 + threadIdx.x < b.total_aa) {
        const AaTexel x(b, w0 + threadIdx.x);
        const Grid g = x.grid();
        const float4 c = ld_texel(g.lp, g.fmt, x.t);
        edge = !Cross(g, x.c, x.j, RowDiv(x.n), x.t).flat();
        if (!edge) x.store(c);
    }
    const unsigned m = __ballot_sync(0xffffffffu, edge);
    int at = 0;
    if (lane == 0 && m) at = atomicAdd(&n_edges, __popc(m));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (edge) edges[at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)threadIdx.x;
    __syncthreads();
    if ((int)threadIdx.x < n_edges) {
        const AaTexel x(b, w0 + edges[threadIdx.x]);
        x.store(fxaa_edge(x.grid(), x.c, x.j, x.n, x.t));
    }
}
}  // namespace

template <class B>
cudaError_t launch_fxaa(const B& b, cudaStream_t s) {
    if (b.total_aa <= 0) return cudaSuccess;
    int cols = 0;
    for (int k = 0; k < b.n; ++k) cols = max(cols, b.d[k].n_cols);
    const unsigned filters = (unsigned)((b.total_aa + kFilterThreads - 1) / kFilterThreads);
    const cudaError_t e = launch_overlapped(k_lp_luma<B>, dim3(cols, kLumaParts, b.n), kLumaThreads, 0, s, b);
    if (e != cudaSuccess) return e;
    return launch_overlapped(k_fxaa_lp<B>, filters, kFilterThreads, 0, s, b);
}

template cudaError_t launch_fxaa<SmallBatch>(const SmallBatch&, cudaStream_t);
template cudaError_t launch_fxaa<BigBatch>(const BigBatch&, cudaStream_t);

}  // namespace vafr
