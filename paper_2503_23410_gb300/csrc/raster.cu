// raster.cu -- the deferred pipeline (Sec. 3.4, Sec. 5): a visibility buffer
// rasterised at display resolution whose coverage test is the GT cast's, and
// lighting from it in the LP buffer or at every pixel.
#include "trace.cuh"

#include <limits.h>

namespace vafr {
namespace {

// ---- deferred path (Sec. 3.4 / Sec. 5: G-buffer at native resolution, lighting
// in the LP buffer) ------------------------------------------------------------
// The G-buffer is a visibility buffer: per display pixel the 64-bit key
// (hit distance bits << 32) | triangle id of the closest triangle, written by
// a rasteriser whose coverage test is the watertight test of the pixel-centre
// ray (so the buffer equals the GT cast's closest hits exactly); the LP pass
// shades each texel from the pixel under its screen point, the GT pass every
// pixel.

constexpr float kClipZ = 1e-4f;       // camera-space near plane for bounding boxes

__device__ __forceinline__ void pixel_ray(const FrameDesc& f, int x, int y, Ray& r) {
    const float cx = f.cr * ((float)x + 0.5f - 0.5f * (float)f.W);
    const float cy = f.cr * (0.5f * (float)f.H - ((float)y + 0.5f));
    world_ray(f, cx, cy, r);
}

// Camera coordinates R^T (v - o) of a world point.
__device__ __forceinline__ float3 to_camera(const FrameDesc& f, float4 v) {
    const float x = v.x - f.org[0], y = v.y - f.org[1], z = v.z - f.org[2];
    return make_float3(fmaf(f.R[0], x, fmaf(f.R[3], y, f.R[6] * z)),
                       fmaf(f.R[1], x, fmaf(f.R[4], y, f.R[7] * z)),
                       fmaf(f.R[2], x, fmaf(f.R[5], y, f.R[8] * z)));
}

// Pixel bounding box of a triangle's part inside the view frustum: the
// triangle (camera coordinates) is clipped (Sutherland-Hodgman) by z >= kClipZ
// and by the four side planes |x| <= z hx, |y| <= z hy of the display widened
// by two pixels, then projected; the box is widened by one pixel.  False if
// nothing remains.
__device__ __forceinline__ int clip_poly(const float3* in, int n, float3* out, float px, float py, float pz, float pw) {
    // keeps the points with px x + py y + pz z + pw >= 0
    int m = 0;
    for (int e = 0; e < n; ++e) {
        const float3 a = in[e], b = in[e + 1 == n ? 0 : e + 1];
        const float da = fmaf(px, a.x, fmaf(py, a.y, fmaf(pz, a.z, pw)));
        const float db = fmaf(px, b.x, fmaf(py, b.y, fmaf(pz, b.z, pw)));
        if (da >= 0.0f) out[m++] = a;
        if ((da >= 0.0f) != (db >= 0.0f)) {
            const float s = da / (da - db);
            out[m++] = make_float3(fmaf(s, b.x - a.x, a.x), fmaf(s, b.y - a.y, a.y), fmaf(s, b.z - a.z, a.z));
        }
    }
    return m;
}

__device__ __forceinline__ bool tri_bbox(const FrameDesc& f, float3 p[3], int& x0, int& y0, int& x1, int& y1) {
    float3 A[8], Bv[8];
    A[0] = p[0]; A[1] = p[1]; A[2] = p[2];
    const float hx = f.cr * (0.5f * (float)f.W + 2.0f), hy = f.cr * (0.5f * (float)f.H + 2.0f);
    // the same five planes on the vertices: all outside one plane -> nothing
    // to draw; all inside every plane -> the vertices are the polygon
    unsigned in_all = 0x1fu, out_any = 0u;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float3 v = p[k];
        const unsigned in = (v.z - kClipZ >= 0.0f ? 1u : 0u) | (fmaf(v.z, hx, -v.x) >= 0.0f ? 2u : 0u) |
                            (fmaf(v.z, hx, v.x) >= 0.0f ? 4u : 0u) | (fmaf(v.z, hy, -v.y) >= 0.0f ? 8u : 0u) |
                            (fmaf(v.z, hy, v.y) >= 0.0f ? 16u : 0u);
        in_all &= in;
        out_any |= in;
    }
    if (out_any != 0x1fu) return false;   // some plane has every vertex outside
    int m;
    if (in_all == 0x1fu) {
        Bv[0] = p[0]; Bv[1] = p[1]; Bv[2] = p[2];
        m = 3;
    } else {
        m = clip_poly(A, 3, Bv, 0.0f, 0.0f, 1.0f, -kClipZ);
        if (m) m = clip_poly(Bv, m, A, -1.0f, 0.0f, hx, 0.0f);
        if (m) m = clip_poly(A, m, Bv, 1.0f, 0.0f, hx, 0.0f);
        if (m) m = clip_poly(Bv, m, A, 0.0f, -1.0f, hy, 0.0f);
        if (m) m = clip_poly(A, m, Bv, 0.0f, 1.0f, hy, 0.0f);
        if (m == 0) return false;
    }
    float lx = INFINITY, ly = INFINITY, hxs = -INFINITY, hys = -INFINITY;
    const float ic = 1.0f / f.cr;
    for (int k = 0; k < m; ++k) {
        const float sx = fmaf(Bv[k].x / Bv[k].z, ic, 0.5f * (float)f.W);
        const float sy = fmaf(-Bv[k].y / Bv[k].z, ic, 0.5f * (float)f.H);
        lx = fminf(lx, sx); hxs = fmaxf(hxs, sx);
        ly = fminf(ly, sy); hys = fmaxf(hys, sy);
    }
    // pixel x covers [x, x + 1): centres in the box, plus a pixel of slack
    const float fx0 = fmaxf(floorf(lx - 0.5f) - 1.0f, 0.0f), fy0 = fmaxf(floorf(ly - 0.5f) - 1.0f, 0.0f);
    const float fx1 = fminf(ceilf(hxs - 0.5f) + 1.0f, (float)(f.W - 1));
    const float fy1 = fminf(ceilf(hys - 0.5f) + 1.0f, (float)(f.H - 1));
    if (!(fx0 <= fx1 && fy0 <= fy1)) return false;
    x0 = (int)fx0; y0 = (int)fy0; x1 = (int)fx1; y1 = (int)fy1;
    return true;
}

// Per-triangle raster set-up: world vertices, id, the camera-depth lower
// bound t_lo of any hit (rays are (cx, cy, 1) in camera space, so a hit's
// distance t is its camera depth), and the screen-space pre-filter.
//
// Pre-filter: the three edge functions of the triangle's projection, scaled
// so each is the signed pixel distance to its edge (positive inside).  A pixel
// whose centre is more than `slack` pixels outside an edge cannot be hit by
// its ray.  The slack bounds the gap between the FP32 projection and the FP32
// watertight test: both err by a few units in the last place of the
// coordinates they handle, which in pixel units is ~2^-24 (|s| + (|v| + |o| +
// |v - o|) / (z_min c_r)) for projected coordinates s, world vertices v, eye o
// and nearest depth z_min; the slack takes 2^-16 times that (256x margin)
// plus 1/64 pixel.  Triangles crossing the near plane, degenerate
// projections, or a slack above 2^16 pixels use no filter.
constexpr float kEdgeSlack = 1.0f / 64.0f;
struct TriSetup {
    float3 A, B, C;           // vertices minus the eye, as the watertight test forms them
    int id;
    float t_lo;               // every hit of the triangle has t >= t_lo
    float ea[3], eb[3], ec[3];  // e_i(x, y) = ea_i x + eb_i y + ec_i
    float slack;
    bool filt;
};

__device__ __forceinline__ float max_abs3(float x, float y, float z) {
    return fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)));
}

__device__ __forceinline__ void tri_setup(const FrameDesc& f, const float4& a, const float4& b, const float4& c,
                                          const float3 p[3], TriSetup& T) {
    T.A = make_float3(__fsub_rn(a.x, f.org[0]), __fsub_rn(a.y, f.org[1]), __fsub_rn(a.z, f.org[2]));
    T.B = make_float3(__fsub_rn(b.x, f.org[0]), __fsub_rn(b.y, f.org[1]), __fsub_rn(b.z, f.org[2]));
    T.C = make_float3(__fsub_rn(c.x, f.org[0]), __fsub_rn(c.y, f.org[1]), __fsub_rn(c.z, f.org[2]));
    T.id = __float_as_int(a.w);
    const float zmin = fminf(p[0].z, fminf(p[1].z, p[2].z));
    const float vmax = fmaxf(max_abs3(a.x, a.y, a.z), fmaxf(max_abs3(b.x, b.y, b.z), max_abs3(c.x, c.y, c.z)));
    const float omax = max_abs3(f.org[0], f.org[1], f.org[2]);
    float dmax = 0.0f;
    for (int k = 0; k < 3; ++k) dmax = fmaxf(dmax, max_abs3(p[k].x, p[k].y, p[k].z));
    // camera depth of a hit is >= zmin; FP32 rounding of depths and of t is
    // far below 2^-12 of the magnitudes involved
    T.t_lo = zmin - ldexpf(fabsf(zmin) + vmax + omax + dmax, -12);
    T.filt = false;
    T.slack = 0.0f;
    if (!(zmin > kClipZ)) return;
    float sx[3], sy[3];
    const float ic = 1.0f / f.cr;
    float M = 0.5f * (float)max(f.W, f.H);
    for (int k = 0; k < 3; ++k) {
        sx[k] = fmaf(p[k].x / p[k].z, ic, 0.5f * (float)f.W);
        sy[k] = fmaf(-p[k].y / p[k].z, ic, 0.5f * (float)f.H);
        M = fmaxf(M, fmaxf(fabsf(sx[k]), fabsf(sy[k])));
    }
    const float area = (sx[1] - sx[0]) * (sy[2] - sy[0]) - (sx[2] - sx[0]) * (sy[1] - sy[0]);
    T.slack = kEdgeSlack + ldexpf(M + (vmax + omax + dmax) / (zmin * f.cr), -16);
    if (!(isfinite(area) && fabsf(area) > 1e-6f && T.slack < 65536.0f)) return;
    const float sg = area > 0.0f ? 1.0f : -1.0f;
    for (int k = 0; k < 3; ++k) {
        const int q = k == 2 ? 0 : k + 1;
        const float ex = sx[q] - sx[k], ey = sy[q] - sy[k];
        const float inv = sg * rsqrtf(fmaxf(fmaf(ex, ex, ey * ey), 1e-30f));
        // e = (ex (y - sy_k) - ey (x - sx_k)) / |edge|, positive inside
        T.ea[k] = -ey * inv;
        T.eb[k] = ex * inv;
        T.ec[k] = (ey * sx[k] - ex * sy[k]) * inv;
    }
    T.filt = true;
}

// Counters of the instrumented (STATS) rasteriser launch: pre-filter
// evaluations (box pixels outside culled tiles), pixels past the pre-filter,
// exact tests run (past the depth pre-test), atomic minima issued.
struct RasterCounts {
    unsigned long long box_px, filtered, tests, atomics;
};

template <bool STATS>
__device__ __forceinline__ void flush_counts(const RasterCounts& n, unsigned long long* stats) {
    if (!STATS || stats == nullptr) return;
    atomicAdd(stats + 0, n.box_px);
    atomicAdd(stats + 1, n.filtered);
    atomicAdd(stats + 2, n.tests);
    atomicAdd(stats + 3, n.atomics);
}

// Both passes work a warp at a time: 32 triangles are set up side by side, one
// to a lane, into shared-memory slots; then the lanes take the pixels of their
// boxes, or of the tiles left of them, in turn: pre-filter, depth pre-test, and
// what passes both goes into a queue that is tested exactly 32 pixels at a time.
// Of the 88 M box pixels of a 4K frame of the 1.07 M triangle terrain 35 M pass
// the pre-filter and 20 M the depth pre-test (18 M where each is looked at only when
// its turn to be tested has come).  When each warp step ran the exact test (some 150
// instructions) for whichever lanes had passed, and a thread rasterised its own
// small triangle (13 of 32 lanes busy), the visibility buffer took 800 us; it took
// 465 so, and takes 411 since the triangle test shears by axis (1080p 331 -> 239, 8K
// of 2 M triangles 5,430 -> 1,800).  kSteps depths are loaded before any is looked
// at, and the tile pass hands out its work as it goes: with one load at a time and
// equal runs of tiles it took 724 us before that.
constexpr int kSteps = 4;   // pixels that a lane looks at before any is tested
struct RasterWarp {
    float4 e[3][32];          // edge functions (ea, eb, ec, slack): inside where ea x + eb y + ec > -slack
    float4 v[3][32];          // vertices minus the eye: A | id, B | t_lo, C | -
    int4 box[32];             // first and last pixel
    unsigned xy[32 + 32 * kSteps];          // queue: pixel (y << 16 | x) ...
    unsigned char slot[32 + 32 * kSteps];   // ... and slot
};

__device__ __forceinline__ void put_slot(RasterWarp& w, int s, const TriSetup& T, int4 box) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
        w.e[k][s] = T.filt ? make_float4(T.ea[k], T.eb[k], T.ec[k], T.slack) : make_float4(0.0f, 0.0f, 0.0f, 1.0f);
    w.v[0][s] = make_float4(T.A.x, T.A.y, T.A.z, __int_as_float(T.id));
    w.v[1][s] = make_float4(T.B.x, T.B.y, T.B.z, T.t_lo);
    w.v[2][s] = make_float4(T.C.x, T.C.y, T.C.z, 0.0f);
    w.box[s] = box;
}

// Depth of the hit that pixel (x, y) holds: a triangle with no hit nearer than
// that need not be tested (a stale read only costs a test, the keys only
// decrease; sky (~0) reads as NaN, which is not below anything).
__device__ __forceinline__ float stored_depth(const FrameDesc& f, const unsigned long long* vbuf, int x, int y) {
    return __uint_as_float((unsigned)(vbuf[(long long)y * f.W + x] >> 32));
}

// Exact coverage of the queue's last `n` pixels: the pixel ray's watertight
// test and an atomic minimum of the key.
template <bool STATS>
__device__ __forceinline__ void test_queued(const FrameDesc& f, unsigned long long* vbuf, const RasterWarp& w, int end,
                                            int n, RasterCounts& c) {
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const int q = end - n + lane;
        const int x = (int)(w.xy[q] & 0xffffu), y = (int)(w.xy[q] >> 16), s = w.slot[q];
        const float4 A = w.v[0][s], B = w.v[1][s], C = w.v[2][s];
        if (STATS) ++c.tests;
        Ray r;
        pixel_ray(f, x, y, r);
        ray_shear(r);   // the triangle test needs no box data
        const float t = tri_test_rel(r, make_float3(A.x, A.y, A.z), make_float3(B.x, B.y, B.z),
                                     make_float3(C.x, C.y, C.z));
        if (t < INFINITY) {
            unsigned long long* px = vbuf + (long long)y * f.W + x;
            const unsigned long long key =
                ((unsigned long long)__float_as_uint(t) << 32) | (unsigned)__float_as_int(A.w);
            if (key < *px) {
                atomicMin(px, key);
                if (STATS) ++c.atomics;
            }
        }
    }
    __syncwarp();
}

// Appends a lane's pixel if `pass`.
__device__ __forceinline__ void queue_pixel(RasterWarp& w, int& queued, bool pass, int x, int y, int s) {
    const unsigned m = __ballot_sync(0xffffffffu, pass);
    if (pass) {
        const int q = queued + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
        w.xy[q] = (unsigned)y << 16 | (unsigned)x;
        w.slot[q] = (unsigned char)s;
    }
    queued += __popc(m);
}

// Tests the queue 32 pixels at a time until fewer are left (all: none).
template <bool STATS>
__device__ __forceinline__ void drain(const FrameDesc& f, unsigned long long* vbuf, const RasterWarp& w, int& queued,
                                      bool all, RasterCounts& c) {
    __syncwarp();
    while (queued >= 32 || (all && queued > 0)) {
        const int n = min(queued, 32);
        test_queued<STATS>(f, vbuf, w, queued, n, c);
        queued -= n;
    }
}

// Large triangles are split into kTileW x kTileH pixel tiles of their boxes.
// One 64-bit counter hands out (record slot << kTileBits) | first tile, so the
// records' first tiles increase with the slot: the tile pass finds a tile's
// record by binary search.  n_tris < 2^30 bounds the slots; a tile sum that
// would pass 2^kTileBits is reported as a fault.
// Boxes above kSmallTriPixels go to the tile pass: 48, 64, 96 and 128 pixels took
// 505, 474, 465 and 472 us at 4K and 57, 58, 59 and 67 us at 640 x 360 with 60 K
// triangles.
constexpr int kSmallTriPixels = 96;
constexpr int kTileW = 16, kTileH = 8;
constexpr int kTileRows = 32 / kTileW;   // tile rows a warp covers per step
static_assert(32 % kTileW == 0 && kTileH % kTileRows == 0, "tile shape");
constexpr int kTileBits = 34;
constexpr unsigned long long kTileMask = (1ull << kTileBits) - 1;
constexpr int kRasterWarps = 4;    // per block
constexpr int kRasterBlocks = 8;   // per SM

// Pass 1: every triangle is set up; a warp rasterises the small boxes of its
// `per` triangles (at most 32), large ones are recorded for pass 2.
template <bool STATS>
__global__ void __launch_bounds__(32 * kRasterWarps, kRasterBlocks)
k_vbuf_raster(const SceneDev sc, const __grid_constant__ SmallBatch b, unsigned long long* vbuf, int4* big,
              int* big_leaf, long long* big_first, unsigned long long* counter, unsigned big_cap, int per,
              unsigned long long* stats) {
    after_previous();
    __shared__ RasterWarp warps[kRasterWarps];
    __shared__ int starts[kRasterWarps][32];
    __shared__ float widths[kRasterWarps][32];   // 1 / box width
    RasterWarp& w = warps[threadIdx.x >> 5];
    int* start_of = starts[threadIdx.x >> 5];
    float* inv_width = widths[threadIdx.x >> 5];
    const FrameDesc& f = b.d[0];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    RasterCounts n{};
    const int n_warps = (int)gridDim.x * kRasterWarps;
    for (int g = (int)blockIdx.x * kRasterWarps + (int)(threadIdx.x >> 5); (long long)g * per < sc.n_tris;
         g += n_warps) {
        const long long k = lane < per ? (long long)g * per + lane : sc.n_tris;
        int area = 0;
        int4 box = make_int4(0, 0, 0, 0);
        float4 a, bb, c;
        float3 p[3];
        if (k < sc.n_tris) {
            a = __ldg(sc.leaves + 3 * k);
            bb = __ldg(sc.leaves + 3 * k + 1);
            c = __ldg(sc.leaves + 3 * k + 2);
            p[0] = to_camera(f, a);
            p[1] = to_camera(f, bb);
            p[2] = to_camera(f, c);
            // behind the eye, or outside the frustum: nothing to draw
            if (!(p[0].z <= 0.0f && p[1].z <= 0.0f && p[2].z <= 0.0f) &&
                tri_bbox(f, p, box.x, box.y, box.z, box.w)) {
                const int bw = box.z - box.x + 1, bh = box.w - box.y + 1;
                area = bw * bh;
                if (area > kSmallTriPixels) {
                    area = 0;
                    const unsigned long long nt = (unsigned long long)((bw + kTileW - 1) / kTileW) *
                                                  (unsigned long long)((bh + kTileH - 1) / kTileH);
                    const unsigned long long old = atomicAdd(counter, (1ull << kTileBits) | nt);
                    const unsigned long long slot = old >> kTileBits, first = old & kTileMask;
                    if (slot < big_cap && first + nt <= kTileMask) {
                        big[slot] = box;
                        big_leaf[slot] = (int)k;
                        big_first[slot] = (long long)first;
                    } else {
                        atomicOr(f.status, kFaultBadNode);   // list overflow: reported, never silent
                    }
                }
            }
        }
        // the small ones' slots, and where their pixels start
        const unsigned some = __ballot_sync(full, area > 0);
        if (!some) continue;
        const int slots = __popc(some);
        int incl = area;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(full, incl, 31);
        if (area > 0) {
            const int s = __popc(some & lt);
            TriSetup T;
            tri_setup(f, a, bb, c, p, T);
            put_slot(w, s, T, box);
            start_of[s] = incl - area;
            inv_width[s] = 1.0f / (float)(box.z - box.x + 1);
        }
        __syncwarp();
        const int my_start = lane < slots ? start_of[lane] : INT_MAX;
        int queued = 0;
        for (int base = 0; base < total; base += 32 * kSteps) {
            int sl[kSteps], px[kSteps], py[kSteps];
            bool pass[kSteps];
#pragma unroll
            for (int q = 0; q < kSteps; ++q) {
                // the slot of pixel i: the starts in these 32 pixels as bits
                const int from = base + 32 * q, i = from + lane;
                const int at = __popc(__ballot_sync(full, my_start <= from)) - 1;
                const unsigned bits =
                    __reduce_or_sync(full, my_start > from && my_start < from + 32 ? 1u << (my_start - from) : 0u);
                const int s = at + __popc(bits & (lt | 1u << lane));
                sl[q] = s;
                pass[q] = false;
                if (i < total) {
                    const int local = i - start_of[s];
                    const int4 bx = w.box[s];
                    const int row = (int)(((float)local + 0.5f) * inv_width[s]);   // exact: local < 2^10
                    px[q] = bx.x + local - row * (bx.z - bx.x + 1);
                    py[q] = bx.y + row;
                    const float x = (float)px[q] + 0.5f, y = (float)py[q] + 0.5f;
                    const float4 e0 = w.e[0][s], e1 = w.e[1][s], e2 = w.e[2][s];
                    if (STATS) ++n.box_px;
                    pass[q] = fmaf(e0.x, x, fmaf(e0.y, y, e0.z)) > -e0.w && fmaf(e1.x, x, fmaf(e1.y, y, e1.z)) > -e1.w &&
                              fmaf(e2.x, x, fmaf(e2.y, y, e2.z)) > -e2.w;
                    if (STATS && pass[q]) ++n.filtered;
                }
            }
            float depth[kSteps];
#pragma unroll
            for (int q = 0; q < kSteps; ++q) depth[q] = pass[q] ? stored_depth(f, vbuf, px[q], py[q]) : 0.0f;
#pragma unroll
            for (int q = 0; q < kSteps; ++q)
                queue_pixel(w, queued, pass[q] && !(depth[q] < w.v[1][sl[q]].w), px[q], py[q], sl[q]);
            drain<STATS>(f, vbuf, w, queued, false, n);
        }
        drain<STATS>(f, vbuf, w, queued, true, n);
        __syncwarp();   // the slots are reused
    }
    flush_counts<STATS>(n, stats);
}

// Pass 2: warps take 32 consecutive tiles at a time (a counter, as some have far
// more pixels to test than others), set up their triangles, 32 or fewer, try
// the tiles against the edges side by side, and look at the pixels of those that
// remain, kSteps rows pairs of 16 pixels at once.
// Records are checked against the display and the scene before use, so a list
// damaged by an overflow (already reported by pass 1) cannot lead out of bounds.
static_assert(kTileH == kSteps * kTileRows, "a tile is looked at in one go");
template <bool STATS>
__global__ void __launch_bounds__(32 * kRasterWarps, kRasterBlocks)
k_vbuf_tiles(const SceneDev sc, const __grid_constant__ SmallBatch b, unsigned long long* vbuf, const int4* big,
             const int* big_leaf, const long long* big_first, unsigned long long* counter, unsigned big_cap,
             unsigned long long* stats) {
    after_previous();
    __shared__ RasterWarp warps[kRasterWarps];
    RasterWarp& w = warps[threadIdx.x >> 5];
    const FrameDesc& f = b.d[0];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    RasterCounts n{};
    const unsigned long long cnt = counter[0];
    const long long total = (long long)(cnt & kTileMask);
    const long long n_rec = min((long long)(cnt >> kTileBits), (long long)big_cap);
    if (n_rec <= 0) return;
    // 32 tiles at a time, fewer where that would leave warps without any
    const long long n_warps = (long long)gridDim.x * kRasterWarps;
    const int take = (int)min(32ll, (total + n_warps - 1) / n_warps);
    while (true) {
        unsigned long long chunk = 0ull;
        if (lane == 0) chunk = atomicAdd(counter + 1, 1ull);
        chunk = __shfl_sync(full, chunk, 0);
        const long long g = (long long)chunk * take;
        if (g >= total) break;
        const long long end = min(g + take, total);
        // last record whose first tile is <= g, by 32 probes at a time
        long long lo = 0, hi = n_rec;   // in [lo, hi)
        while (hi - lo > 1) {
            const long long step = (hi - lo + 31) / 32;
            const long long at = lo + step * (lane + 1);
            const int below = __popc(__ballot_sync(full, at < hi && big_first[at] <= g));
            lo += step * below;
            hi = min(hi, lo + step);
        }
        // the triangles of these tiles, one to a lane
        const long long rec = lo + lane;
        const long long first = rec < n_rec ? big_first[rec] : LLONG_MAX;
        int ntx = 0, nt = 0;   // tiles per row of the box, tiles; 0: not to be drawn
        if (first < end) {
            const int4 bx = big[rec];
            const int k = big_leaf[rec];
            if (k >= 0 && k < sc.n_tris && bx.x >= 0 && bx.y >= 0 && bx.x <= bx.z && bx.y <= bx.w && bx.z < f.W &&
                bx.w < f.H) {
                const float4 a = __ldg(sc.leaves + 3ll * k), bb = __ldg(sc.leaves + 3ll * k + 1),
                             c = __ldg(sc.leaves + 3ll * k + 2);
                const float3 p[3] = {to_camera(f, a), to_camera(f, bb), to_camera(f, c)};
                TriSetup T;
                tri_setup(f, a, bb, c, p, T);
                put_slot(w, lane, T, bx);
                ntx = (bx.z - bx.x + kTileW) / kTileW;
                nt = ntx * ((bx.w - bx.y + kTileH) / kTileH);   // <= 2^23
            }
        }
        __syncwarp();
        // the slot of tile g + lane: the first tiles as bits
        const unsigned bits = __reduce_or_sync(full, first > g && first < g + 32 ? 1u << (int)(first - g) : 0u);
        const int s = __popc(bits & ((2u << lane) - 1u));
        const long long t = g + lane - __shfl_sync(full, first, s);
        const int across = __shfl_sync(full, ntx, s), tiles = __shfl_sync(full, nt, s);
        bool draw = false;
        int tx = 0, ty = 0;
        if (g + lane < end && t >= 0 && t < tiles) {
            const int4 bx = w.box[s];
            tx = bx.x + ((int)t % across) * kTileW;
            ty = bx.y + ((int)t / across) * kTileH;
            // not wholly outside one edge (at the tile's pixel-centre corner
            // that maximises it, with twice the slack)
            const float cx0 = (float)tx + 0.5f, cx1 = (float)min(tx + kTileW - 1, bx.z) + 0.5f;
            const float cy0 = (float)ty + 0.5f, cy1 = (float)min(ty + kTileH - 1, bx.w) + 0.5f;
            draw = true;
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const float4 v = w.e[e][s];
                draw &= !(fmaf(v.x, v.x > 0.0f ? cx1 : cx0, fmaf(v.y, v.y > 0.0f ? cy1 : cy0, v.z)) <= -2.0f * v.w);
            }
        }
        int queued = 0;
        for (unsigned todo = __ballot_sync(full, draw); todo; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            const int ts = __shfl_sync(full, s, src);
            const int x = __shfl_sync(full, tx, src) + lane % kTileW;
            const int y = __shfl_sync(full, ty, src) + lane / kTileW;
            const int4 bx = w.box[ts];
            const float t_lo = w.v[1][ts].w;
            const float px = (float)x + 0.5f, py = (float)y + 0.5f;
            bool pass[kSteps];
#pragma unroll
            for (int q = 0; q < kSteps; ++q) pass[q] = x <= bx.z && y + kTileRows * q <= bx.w;
            if (STATS)
                for (int q = 0; q < kSteps; ++q) n.box_px += pass[q];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float4 v = w.e[k][ts];
                const float e = fmaf(v.x, px, fmaf(v.y, py, v.z)), slack = -v.w;
#pragma unroll
                for (int q = 0; q < kSteps; ++q) pass[q] = pass[q] && fmaf((float)(kTileRows * q), v.y, e) > slack;
            }
            float depth[kSteps];
#pragma unroll
            for (int q = 0; q < kSteps; ++q) {
                if (STATS) n.filtered += pass[q];
                depth[q] = pass[q] ? stored_depth(f, vbuf, x, y + kTileRows * q) : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < kSteps; ++q)
                queue_pixel(w, queued, pass[q] && !(depth[q] < t_lo), x, y + kTileRows * q, ts);
            drain<STATS>(f, vbuf, w, queued, false, n);
        }
        drain<STATS>(f, vbuf, w, queued, true, n);
        __syncwarp();   // the slots are reused
    }
    flush_counts<STATS>(n, stats);
}

// Shading of display pixel (x, y) from the visibility buffer (the GT cast's
// shading of that pixel: its ray, hit distance and triangle).
__device__ __forceinline__ float4 shade_vbuf(const SceneDev& sc, const FrameDesc& f, const unsigned long long* vbuf,
                                             const int* leaf_of, int x, int y) {
    Ray r;
    pixel_ray(f, x, y, r);
    const unsigned long long key = vbuf[(long long)y * f.W + x];
    Hit h;
    if (key == ~0ull) {
        h.leaf = -1;
        h.id = -1;
        h.t = INFINITY;
    } else {
        h.id = (int)(unsigned)(key & 0xffffffffu);
        h.t = __uint_as_float((unsigned)(key >> 32));
        h.leaf = leaf_of[h.id];
    }
    return shade(sc, r, h);
}

// LP lighting: texel -> the pixel under its screen point (clamped to the
// display) -> that pixel's shading.
__global__ void __launch_bounds__(256)
k_shade_lp_vbuf(const SceneDev sc, const __grid_constant__ SmallBatch b, const unsigned long long* vbuf,
                const int* leaf_of) {
    after_previous();
    const FrameDesc& f = b.d[0];
    for (int k = blockIdx.x * 256 + threadIdx.x; k < f.n_texels; k += gridDim.x * 256) {
        const int2 tc = __ldg(f.work + k);
        const int2 cc = __ldg(&f.col[tc.y]);
        const int j = tc.x - cc.x;
        const float te = __ldg(&f.tan_e[tc.y]);
        float sp, cp;
        sincospif(__fdiv_rn((float)(2 * j + 1), (float)cc.y), &sp, &cp);
        const float cx = fmaf(te, cp, f.gx), cy = fmaf(-te, sp, f.gy);
        const float sx = fmaf(cx, 1.0f / f.cr, 0.5f * (float)f.W), sy = fmaf(-cy, 1.0f / f.cr, 0.5f * (float)f.H);
        const int x = min(max((int)floorf(sx), 0), f.W - 1), y = min(max((int)floorf(sy), 0), f.H - 1);
        const float4 v = shade_vbuf(sc, f, vbuf, leaf_of, x, y);
        store_px(f.lp, tc.x, f.lp_fmt, v);
        if (j == 0) store_px(f.lp, tc.x + cc.y, f.lp_fmt, v);
        if (j == cc.y - 1) store_px(f.lp, tc.x - cc.y, f.lp_fmt, v);
    }
}

// Full-resolution lighting (the deferred GT).
__global__ void __launch_bounds__(256)
k_shade_gt_vbuf(const SceneDev sc, const __grid_constant__ SmallBatch b, const unsigned long long* vbuf,
                const int* leaf_of) {
    after_previous();
    const FrameDesc& f = b.d[0];
    const long long n = (long long)f.W * f.H;
    for (long long p = blockIdx.x * 256ll + threadIdx.x; p < n; p += gridDim.x * 256ll) {
        const int y = (int)(p / f.W), x = (int)(p - (long long)y * f.W);
        store_px(f.disp, p, f.disp_fmt, shade_vbuf(sc, f, vbuf, leaf_of, x, y));
    }
}

__global__ void k_leaf_of(const float4* leaves, int n, int* leaf_of) {
    for (int k = blockIdx.x * 256 + threadIdx.x; k < n; k += gridDim.x * 256)
        leaf_of[__float_as_int(leaves[3ll * k].w)] = k;
}

}  // namespace

cudaError_t launch_vbuffer(const SceneDev& sc, const SmallBatch& b, const VbufScratch& v, cudaStream_t s,
                           int num_sms, unsigned long long* stats) {
    const FrameDesc& f = b.d[0];
    cudaError_t e = cudaMemsetAsync(v.vbuf, 0xff, sizeof(unsigned long long) * (size_t)f.W * f.H, s);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(v.counter, 0, 2 * sizeof(unsigned long long), s)) != cudaSuccess) return e;
    if (sc.n_tris <= 0) return cudaSuccess;
    constexpr int tpb = 32 * kRasterWarps;
    const int blocks = num_sms * kRasterBlocks;   // resident
    // 32 triangles to a warp, fewer where that would leave warps without any
    // (7 K triangles at 1080p: 109 us with 32, 64 with 2); up to four times the
    // resident blocks, as some have far more pixels to test than others (477 us
    // against 506 at 4K with one block in each place)
    const int per = min(32, max(1, (sc.n_tris + blocks * kRasterWarps - 1) / (blocks * kRasterWarps)));
    const int groups = (sc.n_tris + per - 1) / per;
    const int grid = min((groups + kRasterWarps - 1) / kRasterWarps, 4 * blocks);
    if (stats)
        k_vbuf_raster<true><<<grid, tpb, 0, s>>>(sc, b, v.vbuf, v.big, v.big_leaf, v.big_first, v.counter, v.big_cap,
                                                  per, stats);
    else
        k_vbuf_raster<false><<<grid, tpb, 0, s>>>(sc, b, v.vbuf, v.big, v.big_leaf, v.big_first, v.counter, v.big_cap,
                                                   per, nullptr);
    count_launch(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_overlapped(stats ? k_vbuf_tiles<true> : k_vbuf_tiles<false>, (unsigned)blocks, tpb, 0, s, sc, b,
                             v.vbuf, v.big, v.big_leaf, v.big_first, v.counter, v.big_cap, stats);
}

cudaError_t launch_leaf_of(const SceneDev& sc, int* leaf_of, cudaStream_t s, int num_sms) {
    if (sc.n_tris <= 0) return cudaSuccess;
    k_leaf_of<<<(unsigned)min((sc.n_tris + 255) / 256, num_sms * 16), 256, 0, s>>>(sc.leaves, sc.n_tris, leaf_of);
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_shade_vbuf(const SceneDev& sc, const SmallBatch& b, const unsigned long long* vbuf,
                              const int* leaf_of, bool full_res, cudaStream_t s, int num_sms) {
    if (full_res) {
        const long long n = (long long)b.d[0].W * b.d[0].H;
        return launch_overlapped(k_shade_gt_vbuf, (unsigned)min((n + 255) / 256, (long long)num_sms * 16), 256, 0, s,
                                 sc, b, vbuf, leaf_of);
    }
    return launch_overlapped(k_shade_lp_vbuf, (unsigned)min((b.d[0].n_texels + 255) / 256, num_sms * 16), 256, 0, s,
                             sc, b, vbuf, leaf_of);
}

}  // namespace vafr
