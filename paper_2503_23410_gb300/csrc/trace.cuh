// trace.cuh -- the ray-casting core shared by the ray-cast (render.cu),
// path-traced (pathtrace.cu) and deferred (raster.cu) pipelines: rays, the
// robust box and watertight triangle tests, LBVH / 4-wide traversal, shading,
// LP ray generation and LP stores.  Everything is inline (or internal to each
// translation unit), so each pipeline's kernels are compiled on their own.
//
// Traversal: single-triangle leaves.  Each binary node holds both child boxes
// and each 4-wide node four, laid out per axis so the slabs run on paired FP32
// instructions.  Box tests follow Ize 2013 ("Robust BVH Ray Traversal"): slab
// distances (b - o) (1/d) and the far distance scaled by 1 + 2 gamma_3, so no
// box the ray touches is culled by rounding.  Triangle test: Woop, Benthin,
// Wald 2013 ("Watertight Ray/Triangle Intersection"), two-sided, with the
// 2-D edge functions evaluated without FMA contraction so that a shared edge
// gets exactly opposite values in the two neighbouring triangles.
// Hit rule: closest t > 0; equal t -> lower triangle id.
#pragma once

#include "vafr_internal.cuh"

#include <float.h>
#include <limits.h>

namespace vafr {
namespace {

constexpr float kAmbient = 0.1f;
constexpr float kFarScale = 1.0000003576278687f;   // 1 + 2 gamma_3 in FP32 (gamma_3 = 3u/(1-3u))
constexpr float kDirEps = 1e-30f;

struct Ray {
    float ox, oy, oz;
    float dx, dy, dz;
    float ix, iy, iz;            // 1/d with zero components clamped (box tests only)
    int nx, ny, nz;              // float4 index of each axis's near plane in a 4-wide node
    int kz;                      // the direction's largest axis, and the shear along it:
    float sx, sy, sz;            // -d_kx / d_kz, -d_ky / d_kz, 1 / d_kz; kx, ky follow kz
    int skip;                    // triangle id the ray ignores (the surface it leaves), or -1
};

__device__ __forceinline__ float safe_inv(float d) {
    if (fabsf(d) < kDirEps) d = copysignf(kDirEps, d);
    return 1.0f / d;
}

// The triangle test's part of a ray.  (Woop et al. exchange kx and ky where d_kz < 0
// to keep the winding; the test here is two-sided, and the exchange negates all of
// its terms exactly.)
__device__ __forceinline__ void ray_shear(Ray& r) {
    const float ax = fabsf(r.dx), ay = fabsf(r.dy), az = fabsf(r.dz);
    r.kz = (ax >= ay && ax >= az) ? 0 : (ay >= az ? 1 : 2);
    const float dz = r.kz == 0 ? r.dx : (r.kz == 1 ? r.dy : r.dz);
    const float dx = r.kz == 0 ? r.dy : (r.kz == 1 ? r.dz : r.dx);
    const float dy = r.kz == 0 ? r.dz : (r.kz == 1 ? r.dx : r.dy);
    r.sx = -(dx / dz);
    r.sy = -(dy / dz);
    r.sz = 1.0f / dz;
}

__device__ __forceinline__ void ray_setup(Ray& r) {
    r.ix = safe_inv(r.dx);
    r.iy = safe_inv(r.dy);
    r.iz = safe_inv(r.dz);
    // a 4-wide node stores lo, hi, hi, lo per axis: (near, far) is (hi, lo)
    // from the axis's third float4 when 1/d < 0, (lo, hi) from its first otherwise
    r.nx = r.ix < 0.0f ? 2 : 0;
    r.ny = r.iy < 0.0f ? 6 : 4;
    r.nz = r.iz < 0.0f ? 10 : 8;
    ray_shear(r);
}

// Both child boxes of a node at once (paired FP32).  Slab distances are
// (b - o) (1/d) as in Ize 2013 ("Robust BVH Ray Traversal"): the subtraction
// keeps the sign of b - o exact even for rays parallel to an axis, and the far
// end is scaled by 1 + 2 gamma_3 so a box the ray touches is never culled by
// rounding.  Returns the entry distances (left, right), +inf for a miss.
__device__ __forceinline__ float2 sub2(float a, float b, float o) {
    return __fadd2_rn(make_float2(a, b), make_float2(-o, -o));
}

__device__ __forceinline__ float2 slab2(float4 nx, float4 ny, float4 nz, const Ray& r, float tmax) {
    const float2 ix = make_float2(r.ix, r.ix), iy = make_float2(r.iy, r.iy), iz = make_float2(r.iz, r.iz);
    const float2 x0 = __fmul2_rn(sub2(nx.x, nx.y, r.ox), ix), x1 = __fmul2_rn(sub2(nx.z, nx.w, r.ox), ix);
    const float2 y0 = __fmul2_rn(sub2(ny.x, ny.y, r.oy), iy), y1 = __fmul2_rn(sub2(ny.z, ny.w, r.oy), iy);
    const float2 z0 = __fmul2_rn(sub2(nz.x, nz.y, r.oz), iz), z1 = __fmul2_rn(sub2(nz.z, nz.w, r.oz), iz);
    const float tnl = fmaxf(fmaxf(fminf(x0.x, x1.x), fminf(y0.x, y1.x)), fmaxf(fminf(z0.x, z1.x), 0.0f));
    const float tnr = fmaxf(fmaxf(fminf(x0.y, x1.y), fminf(y0.y, y1.y)), fmaxf(fminf(z0.y, z1.y), 0.0f));
    const float tfl = fminf(fminf(fmaxf(x0.x, x1.x), fmaxf(y0.x, y1.x)), fminf(fmaxf(z0.x, z1.x), tmax));
    const float tfr = fminf(fminf(fmaxf(x0.y, x1.y), fmaxf(y0.y, y1.y)), fminf(fmaxf(z0.y, z1.y), tmax));
    return make_float2(tnl <= tfl * kFarScale ? tnl : INFINITY, tnr <= tfr * kFarScale ? tnr : INFINITY);
}

// Two float4 from one 32-byte aligned address (one 256-bit load).
__device__ __forceinline__ void ldg256(const float4* p, float4& a, float4& b) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}

// Three-input FP32 minimum / maximum (one PTX instruction on sm_100 and later;
// same NaN rule as fminf / fmaxf).
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// max(a, b, c, 0), NaN if the largest is a NaN: as integers, the non-negative
// floats keep their order and the negative ones lie below zero.
__device__ __forceinline__ float max30f(float a, float b, float c) {
    return __int_as_float(__vimax3_s32_relu(__float_as_int(a), __float_as_int(b), __float_as_int(c)));
}

// Sort key of a hit child: its entry distance t >= 0 as bits without the sign (a
// -0 entry is 0), whose unsigned order is the order of t, with the two low bits
// replaced by the slot q, and the sign bit set for an internal child: leaves sort
// before internal children.  `word` is the node's: q for a leaf, kInner | q for
// an internal child, all ones for an unused slot.  Dropping two bits of t only
// reorders children whose distances agree within 4 ulp, and a stack entry's
// distance, rounded down, only culls later.
__device__ __forceinline__ unsigned child_key(float t, unsigned word) {
    return (__float_as_uint(t) & 0x7ffffffcu) | word;
}

// The largest key of an internal child that a ray with closest hit t has to visit:
// t scaled like a box's far end, and finite (a miss is never within it).
__device__ __forceinline__ unsigned key_limit(float t) {
    return __float_as_uint(fminf(t * kFarScale, FLT_MAX)) | kInner | 3u;
}

// The four child boxes of a 4-wide node (two pairs of paired-FP32 slabs), with
// the same robust evaluation as slab2.  Each axis's near and far planes are
// chosen per ray by the sign of 1/d (the near plane of every box is then its
// lo side, or its hi side, for all four children at once), so each child needs
// only the max of three near distances and the min of three far ones.  The
// node stores each axis as lo, hi, hi, lo: the ray's (near, far) pair is one
// 256-bit load at a 32-byte offset fixed per ray.
// A child is hit when it is entered no later than it is left and, with LIM, than
// the limit (a key_limit); key: the children's sort keys (child_key), all ones for
// a miss.
template <bool LIM>
__device__ __forceinline__ void slab4(const float4* __restrict__ nd, const Ray& r, const uint4& word, unsigned lim,
                                      unsigned key[4]) {
    float4 nxp, fxp, nyp, fyp, nzp, fzp;
    ldg256(nd + r.nx, nxp, fxp);
    ldg256(nd + r.ny, nyp, fyp);
    ldg256(nd + r.nz, nzp, fzp);
    const float2 ix = make_float2(r.ix, r.ix), iy = make_float2(r.iy, r.iy), iz = make_float2(r.iz, r.iz);
    const float2 xna = __fmul2_rn(sub2(nxp.x, nxp.y, r.ox), ix), xnb = __fmul2_rn(sub2(nxp.z, nxp.w, r.ox), ix);
    const float2 xfa = __fmul2_rn(sub2(fxp.x, fxp.y, r.ox), ix), xfb = __fmul2_rn(sub2(fxp.z, fxp.w, r.ox), ix);
    const float2 yna = __fmul2_rn(sub2(nyp.x, nyp.y, r.oy), iy), ynb = __fmul2_rn(sub2(nyp.z, nyp.w, r.oy), iy);
    const float2 yfa = __fmul2_rn(sub2(fyp.x, fyp.y, r.oy), iy), yfb = __fmul2_rn(sub2(fyp.z, fyp.w, r.oy), iy);
    const float2 zna = __fmul2_rn(sub2(nzp.x, nzp.y, r.oz), iz), znb = __fmul2_rn(sub2(nzp.z, nzp.w, r.oz), iz);
    const float2 zfa = __fmul2_rn(sub2(fzp.x, fzp.y, r.oz), iz), zfb = __fmul2_rn(sub2(fzp.z, fzp.w, r.oz), iz);
    const float lf = __uint_as_float(lim & ~kInner);
#define VAFR_CHILD(Q, XN, XF, YN, YF, ZN, ZF, W)                                  \
    {                                                                             \
        const float tn = max30f(XN, YN, ZN);                                      \
        float tf = min3f(XF, YF, ZF) * kFarScale;                                 \
        if (LIM) tf = fminf(tf, lf);                                              \
        key[Q] = tn <= tf ? child_key(tn, W) : ~0u;                               \
    }
    VAFR_CHILD(0, xna.x, xfa.x, yna.x, yfa.x, zna.x, zfa.x, word.x)
    VAFR_CHILD(1, xna.y, xfa.y, yna.y, yfa.y, zna.y, zfa.y, word.y)
    VAFR_CHILD(2, xnb.x, xfb.x, ynb.x, yfb.x, znb.x, zfb.x, word.z)
    VAFR_CHILD(3, xnb.y, xfb.y, ynb.y, yfb.y, znb.y, zfb.y, word.w)
#undef VAFR_CHILD
}

// A vertex (minus the origin) sheared: x', y', and the coordinate along kz.  Each x'
// and y' is rounded as the sum over the axes 2, 1, 0 of a 3 x 3 shear matrix is:
// one FMA where the axis follows kz, a product and a sum where it comes before.
template <int KZ>
__device__ __forceinline__ float3 sheared(const Ray& r, float x, float y, float z) {
    if (KZ == 0) return make_float3(fmaf(r.sx, x, y), fmaf(r.sy, x, z), x);
    if (KZ == 1) return make_float3(fmaf(r.sx, y, z), __fadd_rn(x, __fmul_rn(r.sy, y)), y);
    return make_float3(__fadd_rn(x, __fmul_rn(r.sx, z)), __fadd_rn(y, __fmul_rn(r.sy, z)), z);
}

// Watertight test on the vertices minus the origin; returns t or +inf.  The lanes of a
// warp mostly share kz, so a branch on it costs less than a shear by a matrix of
// zeros and ones per ray (27 instead of 9 to 15 instructions, 9 registers for 4):
// 4K visibility buffer and shading of 1.07 M triangles 510 -> 460 us, 1440p GT 305 ->
// 294, 1,024 triangles at 512 x 512 426 -> 419, 4K cast 154 -> 152.
__device__ __forceinline__ float tri_test_rel(const Ray& r, float3 a, float3 b, float3 c) {
    float3 A, B, C;
    if (r.kz == 2) {
        A = sheared<2>(r, a.x, a.y, a.z);
        B = sheared<2>(r, b.x, b.y, b.z);
        C = sheared<2>(r, c.x, c.y, c.z);
    } else if (r.kz == 1) {
        A = sheared<1>(r, a.x, a.y, a.z);
        B = sheared<1>(r, b.x, b.y, b.z);
        C = sheared<1>(r, c.x, c.y, c.z);
    } else {
        A = sheared<0>(r, a.x, a.y, a.z);
        B = sheared<0>(r, b.x, b.y, b.z);
        C = sheared<0>(r, c.x, c.y, c.z);
    }
    const float U = __fsub_rn(__fmul_rn(C.x, B.y), __fmul_rn(C.y, B.x));
    const float V = __fsub_rn(__fmul_rn(A.x, C.y), __fmul_rn(A.y, C.x));
    const float W = __fsub_rn(__fmul_rn(B.x, A.y), __fmul_rn(B.y, A.x));
    if (min3f(U, V, W) < 0.0f && max3f(U, V, W) > 0.0f) return INFINITY;
    const float det = __fadd_rn(__fadd_rn(U, V), W);
    if (det == 0.0f) return INFINITY;
    const float T = fmaf(U, __fmul_rn(r.sz, A.z), fmaf(V, __fmul_rn(r.sz, B.z), __fmul_rn(W, __fmul_rn(r.sz, C.z))));
    const float t = __fdiv_rn(T, det);
    return t > 0.0f ? t : INFINITY;
}

__device__ __forceinline__ float tri_test(const Ray& r, float4 a, float4 b, float4 c) {
    return tri_test_rel(r, make_float3(__fsub_rn(a.x, r.ox), __fsub_rn(a.y, r.oy), __fsub_rn(a.z, r.oz)),
                        make_float3(__fsub_rn(b.x, r.ox), __fsub_rn(b.y, r.oy), __fsub_rn(b.z, r.oz)),
                        make_float3(__fsub_rn(c.x, r.ox), __fsub_rn(c.y, r.oy), __fsub_rn(c.z, r.oz)));
}

struct Hit {
    float t;
    int leaf;   // sorted leaf index, -1 = miss
    int id;     // triangle id
};

template <bool STATS, bool SKIP = false>
__device__ __forceinline__ void test_leaf(const SceneDev& sc, const Ray& r, int k, Hit& h,
                                          unsigned long long* tri_tests) {
    const float4 a = __ldg(sc.leaves + 3ll * k);
    const float4 b = __ldg(sc.leaves + 3ll * k + 1);
    const float4 c = __ldg(sc.leaves + 3ll * k + 2);
    if (STATS) ++*tri_tests;
    const float t = tri_test(r, a, b, c);
    const int id = __float_as_int(a.w);
    if (SKIP && id == r.skip) return;
    if (t < h.t || (t == h.t && t < INFINITY && id < h.id)) {
        h.t = t;
        h.leaf = k;
        h.id = id;
    }
}

// Closest hit through the binary LBVH.  Returns a fault bit (0 = fine).
template <bool STATS>
__device__ unsigned traverse2(const SceneDev& sc, const Ray& r, Hit& h,
                              unsigned long long* node_visits, unsigned long long* box_tests,
                              unsigned long long* tri_tests) {
    h.t = INFINITY;
    h.leaf = -1;
    h.id = INT_MAX;
    if (sc.n_tris <= 0) return 0u;
    if (sc.root < 0) {   // single triangle
        test_leaf<STATS>(sc, r, 0, h, tri_tests);
        return 0u;
    }
    int stack[kStackSize];
    float stack_t[kStackSize];
    int sp = 0;
    int node = sc.root;
    const int n_inner = sc.n_tris - 1;
    unsigned budget = 4u * (unsigned)sc.n_tris + 64u;
    while (true) {
        if (--budget == 0u) return kFaultWatchdog;
        if ((unsigned)node >= (unsigned)n_inner) return kFaultBadNode;
        if (STATS) { ++*node_visits; *box_tests += 2; }
        const float4* nd = sc.nodes + 4ll * node;
        const float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
        const int cl = __float_as_int(n3.x), cr = __float_as_int(n3.y);
        const float2 tt = slab2(n0, n1, n2, r, h.t);
        float tl = tt.x, tr = tt.y;
        if (tl < INFINITY && cl < 0) {
            if ((unsigned)~cl >= (unsigned)sc.n_tris) return kFaultBadNode;
            test_leaf<STATS>(sc, r, ~cl, h, tri_tests);
            tl = INFINITY;
        }
        if (tr < INFINITY && cr < 0) {
            if ((unsigned)~cr >= (unsigned)sc.n_tris) return kFaultBadNode;
            test_leaf<STATS>(sc, r, ~cr, h, tri_tests);
            tr = INFINITY;
        }
        const bool hl = tl < INFINITY, hr = tr < INFINITY;
        if (hl && hr) {
            if (sp >= kStackSize) return kFaultStack;
            const bool left_first = tl <= tr;
            stack[sp] = left_first ? cr : cl;
            stack_t[sp] = left_first ? tr : tl;
            ++sp;
            node = left_first ? cl : cr;
        } else if (hl) {
            node = cl;
        } else if (hr) {
            node = cr;
        } else {
            // pop, skipping entries that start beyond the current closest hit
            while (true) {
                if (sp == 0) return 0u;
                --sp;
                if (stack_t[sp] <= h.t * kFarScale) break;
            }
            node = stack[sp];
        }
    }
}

// Ascending order of two sort keys (one integer minimum and one maximum).
__device__ __forceinline__ void sort2(unsigned& a, unsigned& b) {
    const unsigned lo = min(a, b);
    b = max(a, b);
    a = lo;
}

// The same as signed numbers.
__device__ __forceinline__ void sort2s(unsigned& a, unsigned& b) {
    const int lo = min((int)a, (int)b);
    b = (unsigned)max((int)a, (int)b);
    a = (unsigned)lo;
}

// Byte q all ones or zero as the sign bit of argument q.
__device__ __forceinline__ unsigned signs(unsigned a, unsigned b, unsigned c, unsigned d) {
    unsigned x, y, z;
    asm("prmt.b32 %0, %1, %2, 0x00fb;" : "=r"(x) : "r"(a), "r"(b));
    asm("prmt.b32 %0, %1, %2, 0xfb00;" : "=r"(y) : "r"(c), "r"(d));
    asm("prmt.b32 %0, %1, %2, 0x7610;" : "=r"(z) : "r"(x), "r"(y));
    return z;
}

// Closest hit through the 4-wide tree: test the four child boxes, test the
// leaf children that were hit, then continue with the nearest internal child
// and push the others far-to-near.  Children are ordered by integer keys (entry
// distance bits and slot); internal children are consecutive nodes, so the slot
// in a key's low bits gives the child's index.  One loop takes the hit leaves of
// a node, so a warp runs as many triangle tests per node as its busiest lane
// needs (not one pass per child slot that any lane needs); the closest-hit rule
// (t, then id) makes the result independent of the order.
//
// ORDER 0 sorts all four keys.  The leaves come first, so the loop takes the
// nearest first and passes over those beyond the closest hit, and the box tests
// need not look at that hit at all.  ORDER 1 only finds the nearest internal child;
// the box tests drop what lies beyond the closest hit, and the loop takes the
// leaves from a mask of the keys' signs: shorter chains from a node to its
// triangles, which small scenes of large overlapping triangles want (their time is
// that of the longest ray).
//
// The kernels that call this issue on 70 % of the cycles, with the ALU pipe (minima,
// comparisons, selections, logic) 60 % busy and the FMA pipe 24 %, so what counts
// is the ALU's work per node.  A miss is a key of all ones rather than an
// infinite distance compared again, the closest hit drops internal children
// through the limit that the keys are compared with anyway, and a stack entry is
// the key as it is.  With infinite distances and references looked at per child
// the 4K cast of 1.07 M triangles took 175 us, now 156; 1440p GT 345, now 305; both
// 8K eyes of 2 M triangles 734, now 680; ORDER 1 on 1,024 triangles at 512 x 512 470,
// now 426.  Where both orders were measured: terrains of 4,800 to 180,000
// triangles 105 to 157 us with ORDER 0, 109 to 168 with 1; soups of 1,024 325 to 807
// with 0, 295 to 760 with 1.
// Returns a fault bit (0 = fine).
// `any`: an occlusion query, which ends at the first hit found.
template <bool STATS, int ORDER, bool SKIP = false>
__device__ __forceinline__ unsigned traverse4(const SceneDev& sc, const Ray& r, Hit& h,
                                              unsigned long long* node_visits, unsigned long long* box_tests,
                                              unsigned long long* tri_tests, bool any = false) {
    h.t = INFINITY;
    h.leaf = -1;
    h.id = INT_MAX;
    if (sc.n_tris <= 0) return 0u;
    if (sc.root < 0) {   // single triangle
        test_leaf<STATS, SKIP>(sc, r, 0, h, tri_tests);
        return 0u;
    }
    unsigned long long stack[kStackSize];
    int sp = 0;
    int node = 0;
    unsigned lim = key_limit(INFINITY);
    unsigned budget = 4u * (unsigned)sc.n_tris + 64u;
    while (true) {
        if (--budget == 0u) return kFaultWatchdog;
        if ((unsigned)node >= (unsigned)sc.n_nodes4) return kFaultBadNode;   // the nodes are allocated at their count
        const float4* nd = sc.nodes4 + 16ll * node;
        float4 rf, kwf;
        ldg256(nd + 12, rf, kwf);
        const uint4 kw = make_uint4(__float_as_uint(kwf.x), __float_as_uint(kwf.y), __float_as_uint(kwf.z),
                                    __float_as_uint(kwf.w));
        const int c0 = __float_as_int(rf.x), c1 = __float_as_int(rf.y), c2 = __float_as_int(rf.z),
                  c3 = __float_as_int(rf.w);
        unsigned k[4];
        slab4<ORDER != 0>(nd, r, kw, lim, k);
        if (STATS) {
            ++*node_visits;
            *box_tests += (c0 != kEmptyRef) + (c1 != kEmptyRef) + (c2 != kEmptyRef) + (c3 != kEmptyRef);
        }
        unsigned k0 = k[0], k1 = k[1], k2 = k[2], k3 = k[3];
        if (ORDER == 0) {
            // ascending: sorting network (0,1) (2,3) (0,2) (1,3) (1,2)
            sort2(k0, k1);
            sort2(k2, k3);
            sort2(k0, k2);
            sort2(k1, k3);
            sort2(k1, k2);
            // the leaves, nearest first; what is left are the internal children
            while (k0 < kInner) {
                if ((k0 | kInner) <= lim) {
                    const int C = k0 & 2u ? (k0 & 1u ? c3 : c2) : (k0 & 1u ? c1 : c0);
                    if ((unsigned)~C >= (unsigned)sc.n_tris) return kFaultBadNode;
                    test_leaf<STATS, SKIP>(sc, r, ~C, h, tri_tests);
                    if (any && h.leaf >= 0) return 0u;
                    lim = key_limit(h.t);
                }
                k0 = k1;
                k1 = k2;
                k2 = k3;
                k3 = ~0u;
            }
        } else {
            unsigned lm = ~signs(k0, k1, k2, k3) & 0x80808080u;
            if (lm) {
                do {
                    const int C = lm & 0x80u ? c0 : (lm & 0x8000u ? c1 : (lm & 0x800000u ? c2 : c3));
                    lm &= lm - 1u;
                    if ((unsigned)~C >= (unsigned)sc.n_tris) return kFaultBadNode;
                    test_leaf<STATS, SKIP>(sc, r, ~C, h, tri_tests);
                } while (lm);
                if (any && h.leaf >= 0) return 0u;
                lim = key_limit(h.t);
            }
            sort2s(k0, k1);
            sort2s(k2, k3);
            sort2s(k0, k2);
            // (as signed numbers internal children come first, and misses and leaves are past the limit)
        }
        unsigned long long e = ((unsigned long long)k0 << 32) | (unsigned)c0;
#define VAFR_IN(K) (ORDER == 0 ? K <= lim : (int)K <= (int)lim)
        if (VAFR_IN(k0)) {
            // a stack entry: the child's key high, its node's first child low
#define VAFR_PUSH(K)                                                                      \
            if (VAFR_IN(K)) {                                                             \
                if (sp >= kStackSize) return kFaultStack;                                 \
                stack[sp++] = ((unsigned long long)K << 32) | (unsigned)c0;               \
            }
            VAFR_PUSH(k3)
            VAFR_PUSH(k2)
            VAFR_PUSH(k1)
#undef VAFR_PUSH
        } else {
            // pop, skipping entries that start beyond the current closest hit
            do {
                if (sp == 0) return 0u;
                e = stack[--sp];
            } while ((unsigned)(e >> 32) > lim);
        }
#undef VAFR_IN
        node = (int)(unsigned)e + (int)((unsigned)(e >> 32) & 3u);
    }
}

// WIDE: 4 (4-wide PLOC tree) or 2 (binary LBVH); ORDER as traverse4's.
template <int WIDE, bool STATS, int ORDER = 0>
__device__ __forceinline__ unsigned traverse(const SceneDev& sc, const Ray& r, Hit& h,
                                             unsigned long long* nv, unsigned long long* bt,
                                             unsigned long long* tt) {
    if (WIDE == 4) return traverse4<STATS, ORDER>(sc, r, h, nv, bt, tt);
    return traverse2<STATS>(sc, r, h, nv, bt, tt);
}

// Unshadowed inverse-square point lights added to acc: rgb max(0, n . l) / |x - p|^2
// for each light at x, hit point p.  Kept out of line so that scenes without
// point lights run the traversal kernels' code unchanged.
__device__ __noinline__ float3 point_lights(const float4* plights, int n, float px, float py, float pz, float nx,
                                            float ny, float nz, float3 acc) {
    for (int q = 0; q < n; ++q) {
        const float4 lp = __ldg(plights + 2 * q), lc = __ldg(plights + 2 * q + 1);
        const float lx = lp.x - px, ly = lp.y - py, lz = lp.z - pz;
        const float d2 = fmaf(lx, lx, fmaf(ly, ly, lz * lz));
        const float c = fmaf(nx, lx, fmaf(ny, ly, nz * lz)) * rsqrtf(d2);
        if (c > 0.0f) {
            const float g = c / d2;
            acc.x = fmaf(lc.x, g, acc.x);
            acc.y = fmaf(lc.y, g, acc.y);
            acc.z = fmaf(lc.z, g, acc.z);
        }
    }
    return acc;
}

__device__ __forceinline__ float4 shade(const SceneDev& sc, const Ray& r, const Hit& h) {
    if (h.leaf < 0) {
        const float inv = rsqrtf(fmaf(r.dx, r.dx, fmaf(r.dy, r.dy, r.dz * r.dz)));
        const float s = 0.5f * fmaf(r.dy, inv, 1.0f);
        return make_float4(1.0f - 0.5f * s, 1.0f - 0.3f * s, 1.0f, 1.0f);
    }
    const float4 a = __ldg(sc.leaves + 3ll * h.leaf);
    const float4 b = __ldg(sc.leaves + 3ll * h.leaf + 1);
    const float4 c = __ldg(sc.leaves + 3ll * h.leaf + 2);
    const float e1x = b.x - a.x, e1y = b.y - a.y, e1z = b.z - a.z;
    const float e2x = c.x - a.x, e2y = c.y - a.y, e2z = c.z - a.z;
    float nx = e1y * e2z - e1z * e2y;
    float ny = e1z * e2x - e1x * e2z;
    float nz = e1x * e2y - e1y * e2x;
    const float inv = rsqrtf(fmaf(nx, nx, fmaf(ny, ny, nz * nz)));
    nx *= inv; ny *= inv; nz *= inv;
    if (fmaf(nx, r.dx, fmaf(ny, r.dy, nz * r.dz)) > 0.0f) { nx = -nx; ny = -ny; nz = -nz; }
    const float lam = fmaxf(0.0f, -fmaf(nx, sc.light[0], fmaf(ny, sc.light[1], nz * sc.light[2])));
    const float s = fmaf(1.0f - kAmbient, lam, kAmbient);
    const float4 al = __ldg(sc.albedo + h.id);
    float3 acc = make_float3(s, s, s);
    if (sc.n_plights > 0)
        acc = point_lights(sc.plights, sc.n_plights, fmaf(h.t, r.dx, r.ox), fmaf(h.t, r.dy, r.oy), fmaf(h.t, r.dz, r.oz), nx, ny, nz, acc);
    return make_float4(al.x * acc.x, al.y * acc.y, al.z * acc.z, 1.0f);
}

__device__ __forceinline__ void store_px(void* base, long long idx, int fmt, float4 v) {
    if (fmt == VAFR_FMT_RGBA16F) {
        const __half2 lo = __floats2half2_rn(v.x, v.y), hi = __floats2half2_rn(v.z, v.w);
        uint2 p;
        p.x = *reinterpret_cast<const unsigned*>(&lo);
        p.y = *reinterpret_cast<const unsigned*>(&hi);
        reinterpret_cast<uint2*>(base)[idx] = p;
    } else {
        reinterpret_cast<float4*>(base)[idx] = v;
    }
}

__device__ __forceinline__ void world_ray(const FrameDesc& f, float cx, float cy, Ray& r) {
    // camera direction (cx, cy, 1) -> world
    r.dx = fmaf(f.R[0], cx, fmaf(f.R[1], cy, f.R[2]));
    r.dy = fmaf(f.R[3], cx, fmaf(f.R[4], cy, f.R[5]));
    r.dz = fmaf(f.R[6], cx, fmaf(f.R[7], cy, f.R[8]));
    r.ox = f.org[0];
    r.oy = f.org[1];
    r.oz = f.org[2];
    r.skip = -1;
}

template <class B>
__device__ __forceinline__ int find_frame(const B& b, long long w, bool tiles) {
    int lo = 0, hi = b.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const long long beg = tiles ? b.d[mid].tile_begin : b.d[mid].work_begin;
        if (beg <= w) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// LP ray of a work item, (slot, column) or number k of the frame's list (Eqs. 3,
// 10, 11): work items visit the texels in screen-space Hilbert order; texel t =
// (c, j) sits at distance r = tan(e_c)/c_r from the gaze at angle phi = (j + 0.5)
// 360/n_c, so its camera direction is (tan(e_c) cos(phi) + gx, -tan(e_c) sin(phi) +
// gy, 1).  Returns the texel's slot; `guard_lo` / `guard_hi` get the guard slots that
// copy it (texel n_c - 1 -> slot before the column, texel 0 -> slot after), or -1.
__device__ __forceinline__ int lp_ray(const FrameDesc& f, int2 tc, Ray& r, int& guard_lo, int& guard_hi) {
    const int2 cc = __ldg(&f.col[tc.y]);
    const int j = tc.x - cc.x;
    const float te = __ldg(&f.tan_e[tc.y]);
    float sp, cp;
    sincospif(__fdiv_rn((float)(2 * j + 1), (float)cc.y), &sp, &cp);
    world_ray(f, fmaf(te, cp, f.gx), fmaf(-te, sp, f.gy), r);
    guard_lo = j == cc.y - 1 ? tc.x - cc.y : -1;
    guard_hi = j == 0 ? tc.x + cc.y : -1;
    return tc.x;
}
__device__ __forceinline__ int lp_ray(const FrameDesc& f, int k, Ray& r, int& guard_lo, int& guard_hi) {
    return lp_ray(f, __ldg(f.work + k), r, guard_lo, guard_hi);
}

// Shaded LP texel (and hit id) into its slot and the guard slots that copy it.
__device__ __forceinline__ void store_lp(const FrameDesc& f, int t, int glo, int ghi, float4 c, int id) {
    store_px(f.lp, t, f.lp_fmt, c);
    if (glo >= 0) store_px(f.lp, glo, f.lp_fmt, c);
    if (ghi >= 0) store_px(f.lp, ghi, f.lp_fmt, c);
    if (f.hit_ids) {
        f.hit_ids[t] = id;
        if (glo >= 0) f.hit_ids[glo] = id;
        if (ghi >= 0) f.hit_ids[ghi] = id;
    }
}

}  // namespace
}  // namespace vafr
