// vafr_internal.cuh -- device data layouts and launch interfaces shared by the
// CUDA translation units of libvafr.so (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "../../include/vafr.h"

namespace vafr {

// ---- device status words --------------------------------------------------
enum DeviceFault : unsigned {
    kFaultStack = 1u,     // traversal stack would overflow
    kFaultWatchdog = 2u,  // traversal iteration limit reached
    kFaultBadNode = 4u,   // child reference out of range
};

constexpr int kStackSize = 128;   // entries; a descent pushes at most 3 per 4-wide level above the last: depth <= 43
constexpr int kEmptyRef = (int)0x80000000;   // unused slot of a 4-wide node
constexpr unsigned kInner = 0x80000000u;     // key word of an internal child in slot q: kInner | q; of a leaf: q
constexpr int kMaxSeg = VAFR_MAX_PIVOTS - 1;

// ---- scene (LBVH) in traversal layout ----------------------------------------
// Internal node i (64 B, four float4), children L and R:
//   n[0] = (L.lo.x, R.lo.x, L.hi.x, R.hi.x)
//   n[1] = (L.lo.y, R.lo.y, L.hi.y, R.hi.y)
//   n[2] = (L.lo.z, R.lo.z, L.hi.z, R.hi.z)
//   n[3] = (L ref, R ref, -, -) as int bits; ref >= 0 internal, < 0 leaf ~k
// Leaf k (sorted order): three float4 (v0.xyz | id), (v1.xyz | 0), (v2.xyz | 0).
// 4-wide node j (256 B, sixteen float4): per axis the planes lo, hi, hi, lo of
// children 0..3 (so the (near, far) pair of either ray direction is one
// 32-byte aligned load), then their refs (>= 0 4-wide node, < 0 leaf ~k,
// kEmptyRef unused), then the slot keys (q for an internal child in slot q,
// all ones otherwise), then padding.  Internal children take the first slots
// and consecutive indices (slot q's node = slot 0's + q); leaves follow,
// unused slots last.  4-wide node 0 is the root.
struct SceneDev {
    const float4* nodes;
    const float4* nodes4;
    int n_nodes4;           // 4-wide nodes (the traversal's bound on a child index)
    const float4* leaves;
    const float4* albedo;   // original triangle order (rgb, 0)
    int root;               // 0 (internal), ~0 (single leaf) or INT_MIN (empty)
    int n_tris;
    float light[3];         // unit light travel direction
    unsigned* status;       // device status word
    const float4* plights;  // [2 n_plights]: (position, 0), (rgb, 0) of each point light
    int n_plights;
};

// ---- per session: forward-map table ------------------------------------------
// u - 1/2 as a function of z = tan(e) = c_r r on [0, tan(e_max)] (Eqs. 3, 12):
// kUTable uniform intervals, interval i holding the cubic Hermite piece
// c.x + t (c.y + t (c.z + t c.w)), t in [0, 1]; entry kUTable is the constant
// u(e_max) - 1/2 used for z >= tan(e_max).
constexpr int kUTable = 2048;

// ---- longest-first LP render: per frame-eye state kept from frame to frame ----
// The LP render takes its work in chunks of 32 consecutive work items (one per
// lane of a warp).  While a frame renders, every chunk whose traversal time
// (the slowest lane's clock cycles) is at least twice the previous frame's
// mean is listed, and the next frame renders the listed chunks before all
// others.  Only the order changes: every chunk is still rendered exactly once,
// so the results are those of the plain order.  Without it the slowest chunks,
// wherever they fall in the work order, decide when the launch ends.  The
// state has two halves used alternately (frame parity): the half being read
// holds this frame's list, the other collects the next frame's and, in its
// first frame's state, counts the launch's work; the host clears the collecting
// half's counters before each frame.
struct LptCounters {
    unsigned long long cyc_sum;   // sum of the chunk costs of the frame
    unsigned chunks_done;         // chunks costed
    unsigned hot_count;           // entries of the list
    // work counters of the frame's launch, on a line of their own (next to the others,
    // whose line every listed chunk updates, a 156 us cast takes 161; so, 154)
    alignas(128) unsigned long long work[2];
};
struct LptState {
    LptCounters ctr[2];
    int* hot[2];                  // [capacity] listed chunks
    unsigned char* flag[2];       // [capacity] 1 = listed
    int capacity;                 // chunks the arrays hold
};
constexpr int kLptChunk = 32;

// ---- one frame-eye of work (kernel parameter; filled on the host in FP64,
// rounded to FP32) ------------------------------------------------------------
struct FrameDesc {
    float R[9];             // camera -> world rotation, row-major
    float org[3];           // eye position
    float gx, gy;           // gaze tangent offsets: c_r (x0 - W/2), c_r (H/2 - y0)
    float cr;               // c_r
    float px0, py0;         // c_r (0.5 - W/2), c_r (H/2 - 0.5): GT ray of pixel (0,0)
    int gxi, gyi;           // floor of the gaze point
    float gxf, gyf;         // 0.5 - fractional part of the gaze point
    int W, H;
    int lp_fmt, disp_fmt;
    const float* tan_e;     // device [C] tan(e_c) of the column centres
    const int2* col;        // device [C] (first texel, texel count)
    const int4* col_pair;   // device [-1 .. C-1] (slot, FP32 bits of count) of c and of min(c + 1, C - 1); [-1] = column 0 twice
    const float4* u_tab;    // device [u_n + 1] cubic pieces of u(z)
    const int2* work;       // device [n_texels] (texel, column) in processing order
    int u_n;                // number of pieces
    float u_inv_h;          // u_n / tan(e_max)
    int n_cols;
    int n_texels;
    void* lp;
    void* lp_aa;            // FXAA output (read by reconstruct) or nullptr: no FXAA
    float* luma;            // FXAA scratch: luma of every LP slot
    float* depth;           // hit distance per LP slot (inf on a miss) or nullptr
    void* disp;
    int* hit_ids;
    unsigned* status;
    long long work_begin;   // first global work item (render) of this frame
    long long tile_begin;   // first global tile (reconstruct) of this frame
    long long aa_begin;     // first global FXAA texel of this frame
    LptState* lpt;          // longest-first state | frame parity (bit 0), or nullptr
};

template <int MAXD>
struct Batch {
    int n;
    long long total_work;   // sum of render work items
    long long total_tiles;  // sum of reconstruct tiles
    long long total_aa;     // sum of FXAA texels (frames with lp_aa)
    unsigned long long* work_counter;  // device counters (persistent fetch; [1]: longest-first list)
    FrameDesc d[MAXD];
};

using SmallBatch = Batch<2>;
using BigBatch = Batch<VAFR_MAX_BATCH>;
// kernel parameters (scene + batch) must fit the 32,764-byte parameter space
static_assert(sizeof(BigBatch) + sizeof(SceneDev) <= 32764, "batch too large for kernel params");

// ---- launch interfaces ---------------------------------------------------------
// Render variants: 0 the default rule (below); 1-5 threads
// per block, tree width, child order, register cap; 6 and 7 the longest-first LP
// order (7: the ray regenerated for shading and at most 72 registers, 7 blocks
// per SM), whose GT is variant 4's kernel.
constexpr int kNumRenderVariants = 8;
constexpr int kLptVariant = 6;
constexpr int kLptVariantLean = 7;
// Variant 0, what a session has until it is tuned: the longest-first order for
// a session's LP casts, else the plain order in 64 registers, both with all
// hit children of a node sorted; and in scenes of up to kPlainTris triangles the
// plain order in 72 registers with only the nearest child put first (which
// variant 0 was everywhere).  Measured against that everywhere: the 4K cast of the
// 1.07 M triangle terrain 171 us for 198, its 1440p GT 345 for 385, casts of
// terrains of 7 to 65 K triangles 97 to 142 us for 120 to 166 (since then the
// traversal takes fewer instructions: 152 and 294 us).  In small scenes neither
// pays: the longest-first bookkeeping costs casts of 60 to 90 us 4 to 6 us, and
// sorting changes soups of 500 to 4,000 triangles by -15 to +13 % from scene to
// scene.
// What decides is the scene, not its size; the line lies where the two about even
// out.  At 1024 x 768, us, nearest child first | longest-first (casts) and sorted (GT),
// for two or three scenes of each kind:
//                         casts                                      GT
//   terrain      700      83 74 | 84 75                              49 42 | 49 43
//   triangles  2,700      101 85 | 94 84                             59 54 | 61 53
//              7,000      103 94 | 87 87                             70 62 | 69 66
//             1.07 M      176 173 | 151 144                          128 103 | 104 100
//   soups of   1,000      394 623 | 405 642                          268 254 | 306 261
//   triangles  4,000      1678 3312 | 1406 3273                      1068 1160 | 1010 1237
//   as large  10,000      4551 8589 2038 | 4181 8544 2272            2774 2661 2070 | 2736 2744 2275
//   as the    40,000      14084 21347 9496 | 15401 21275 10478       8050 6348 9267 | 9522 6813 9925
//   scene     80,000      29489 58937 16602 | 24918 50180 17952      16656 16049 16186 | 15344 13960 17322
//   a fifth  100,000      638 862 288 | 511 396 263                  576 695 318 | 552 288 316
// The leaves' overlap does not separate them either: either order may win where the
// boxes' areas add up to 50 or to 10,000 times the scene's.  A session's own choice is
// vafr_session_autotune's; variant 5 puts the nearest child first in scenes of any
// size, within 4 % of the 72-register kernel.
constexpr int kPlainTris = 4096;
// variants that render with a longest-first order in every batch ...
__host__ __device__ constexpr bool is_lpt_variant(int v) { return v == kLptVariant || v == kLptVariantLean; }
// ... and those whose single-session LP casts of n_tris triangles do
__host__ __device__ constexpr bool has_lpt_kernel(int v, int n_tris) {
    return v == 0 ? n_tris > kPlainTris : is_lpt_variant(v);
}
// Reconstruct variants: column-run tiles (0-3), row tiles (4-7) and the
// column-run tile with its LP footprint staged in shared memory (8).
constexpr int kNumReconVariants = 9;

// tile width/height in pixels; pixels per thread along a row (row tiles), or 0
// for a column-run tile (one thread per display column, `th` rows)
struct ReconShape { int tw, th; int px; };
ReconShape recon_shape(int variant);

// Sets the render kernels' attributes for the current device and context; every
// session does (they are kept neither across devices nor across a device reset).
void prepare_render();
template <class B>
cudaError_t launch_render_lp(const SceneDev& scene, const B& batch, int variant,
                             cudaStream_t s, int num_sms);
template <class B>
cudaError_t launch_render_gt(const SceneDev& scene, const B& batch, int variant,
                             cudaStream_t s, int num_sms);
template <class B>
cudaError_t launch_reconstruct(const B& batch, int variant, cudaStream_t s);
// Path-traced LP buffers (pathtrace.cu): one path per texel, `depth` diffuse
// bounces; FrameDesc.hit_ids, when set, receives depth + 2 ints per slot.
// `scratch` holds path_scratch_bytes device bytes of the launch's own where
// path_uses_pool wants the pool, and is NULL for one path per lane.
bool path_uses_pool(long long work, int depth);
size_t path_scratch_bytes(int num_sms);
template <class B>
cudaError_t launch_path_lp(const SceneDev& scene, const B& batch, unsigned long long seed, int depth,
                           void* scratch, cudaStream_t s, int num_sms);
template <class B>
cudaError_t launch_path_gt(const SceneDev& scene, const B& batch, unsigned long long seed, int depth,
                           void* scratch, cudaStream_t s, int num_sms);
// Ray casting of an explicit list of (slot, column) work items whose count
// is read from device memory (render.cu): the reprojection's holes.  The batch's
// work counter has been cleared.
cudaError_t launch_render_list(const SceneDev& scene, const SmallBatch& batch, const unsigned* count,
                               cudaStream_t s, int num_sms);
// VaFR_Rep reprojection (reproject.cu): left frame d[0] (lp, depth) warped into
// right frame d[1] (lp written, holes appended to `holes` / `count`).
struct RepScratch {
    float4* vert;                 // [left texels] (U, F, depth, flags | column) seen from the right eye
    unsigned long long* zbuf;     // [right slots] (depth bits << 32) | triangle id
    int2* holes;                  // [right texels] (slot, column) left uncovered
    unsigned* count;              // number of holes
    int* tri_out;                 // [right slots] winning triangle id / -1, or nullptr
    unsigned long long* work;     // work counter to clear for the hole cast, or nullptr
};
cudaError_t launch_reproject(const SmallBatch& batch, const RepScratch& r, cudaStream_t s, int num_sms);
// Deferred path (raster.cu): visibility buffer of frame d[0] at display
// resolution, then LP or full-resolution lighting from it.
struct VbufScratch {
    unsigned long long* vbuf;   // [H][W] (hit distance bits << 32) | triangle id, ~0 = sky
    int4* big;                  // large triangles' pixel boxes
    int* big_leaf;              // ... their leaves
    long long* big_first;       // ... and first tiles
    unsigned long long* counter;  // [2]: (records << 34) | tiles; chunks of tiles taken
    unsigned big_cap;
};
// stats (device, 4 counters, zeroed by the caller) selects an instrumented
// copy of the rasteriser that counts pre-filter evaluations, pixels past the
// pre-filter, exact tests and atomic minima; nullptr = the plain kernels.
cudaError_t launch_vbuffer(const SceneDev& sc, const SmallBatch& b, const VbufScratch& v, cudaStream_t s,
                           int num_sms, unsigned long long* stats = nullptr);
cudaError_t launch_leaf_of(const SceneDev& sc, int* leaf_of, cudaStream_t s, int num_sms);
cudaError_t launch_shade_vbuf(const SceneDev& sc, const SmallBatch& b, const unsigned long long* vbuf,
                              const int* leaf_of, bool full_res, cudaStream_t s, int num_sms);
// FXAA inside the LP buffer of every frame with lp_aa set (fxaa.cu).
template <class B>
cudaError_t launch_fxaa(const B& batch, cudaStream_t s);
cudaError_t launch_render_stats(const SceneDev& scene, const SmallBatch& batch,
                                unsigned long long* counters, cudaStream_t s, int num_sms);

void count_launch(int k = 1);

// Launches that overlap their start-up: a kernel launched by launch_overlapped is
// put on the SMs while the one before it is finishing, and waits for its results
// at after_previous, before it touches memory.  Worth 1.6 us a launch in the scene
// build's rounds and 2 to 4 between passes: FXAA of one eye 37 -> 33.5 us, the 4K
// reconstruction 35.3 -> 33.3 (back to back), a 1280 x 720 frame of 64 triangles 63.6
// -> 60.4, with FXAA 89.5 -> 83.9, the warped 8K eye 370 -> 362.  (Casts that let the
// next launch in at their start instead of at their end gain nothing more.)
// Such a kernel has begun while the one before it may still write, so memory that
// an earlier launch writes is not constant for the kernel's whole life, as __ldg and
// ld.global.nc require: buffers of the frame (LP texels, lumas, depths, lists of
// work, visibility) are read by plain loads, which stay behind the wait.  __ldg is
// for the scene and for the layout's tables, which no overlapped launch writes.
__device__ __forceinline__ void after_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, unsigned block, size_t shared, cudaStream_t s,
                              const A&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = shared;
    cfg.stream = s;
    cfg.attrs = &attr;
    // plain launches in captured graphs, whose edges are then plain too
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
        cudaGetLastError();
        capture = cudaStreamCaptureStatusActive;
    }
    cfg.numAttrs = capture == cudaStreamCaptureStatusNone ? 1 : 0;
    count_launch(1);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    if (e != cudaSuccess) cudaGetLastError();   // it is returned, not left for a later call
    return e;
}

// Scene build.  All device pointers are owned by the caller.  The steps run in
// this order, and the caller lays their scratch out so that each step's takes
// the place of the earlier ones':
//   lbvh_sort       Morton codes, their order, the sorted leaves (lbvh.cu)
//   tree4_build     traversal tree: PLOC over the sorted leaves, collapsed to
//                   4-wide nodes, which it numbers and counts (tree4.cu;
//                   synchronises `s` to read the count)
//   tree4_pack      ... written to b.nodes4 (16 float4 per node), which the
//                   caller allocates after tree4_build
//   lbvh_hierarchy  binary radix tree over the sorted codes and its bounds
struct LbvhBuffers {
    const float* tris;      // n x 9 input (device)
    const float* albedo;    // n x 3 (device) or nullptr
    int n;
    // what the scene keeps
    uint32_t* codes;        // n  Morton codes, input order
    int32_t* ids;           // n  sorted triangle ids
    float* leaf_box;        // n x 6
    float4* leaves;         // n x 3
    float4* albedo4;        // n
    float4* nodes4;         // n_nodes4 x 16
    int2* child;            // n-1, written by lbvh_hierarchy
    float* node_box;        // (n-1) x 6, written by lbvh_hierarchy
    float4* nodes;          // (n-1) x 4, written by lbvh_hierarchy
    // from lbvh_sort to lbvh_hierarchy
    uint32_t* keys_sorted;  // n
    // within lbvh_sort
    uint32_t* keys_tmp;     // n
    int32_t* ids_tmp;       // n
    unsigned* hist;         // lbvh_hist_elems(n)
    float* part_bounds;     // 6 * 304
    float* scene_bounds;    // 6
    // from lbvh_sort to tree4_build
    float4* clusters;       // n x 2: leaf boxes with their references
    // within lbvh_hierarchy
    int4* links;            // n-1: each internal node's children, the other end of its leaves, its parent
    int32_t* leaf_parent;   // n
    unsigned* flags;        // n: arrival counters of the nodes, then the length of `climbers`
    int32_t* climbers;      // n: children whose parents are made last
};
size_t lbvh_sort_blocks(int n);
size_t lbvh_hist_elems(int n);
cudaError_t lbvh_sort(const LbvhBuffers& b, cudaStream_t s);
cudaError_t lbvh_hierarchy(const LbvhBuffers& b, cudaStream_t s);
// `scratch`: tree4_scratch_bytes(n) device bytes, from tree4_build to tree4_pack.
size_t tree4_scratch_bytes(int n);
cudaError_t tree4_build(const LbvhBuffers& b, void* scratch, cudaStream_t s, int num_sms, int* n_nodes4);
cudaError_t tree4_pack(const LbvhBuffers& b, void* scratch, int n_nodes4, cudaStream_t s);

// FP32 issue rate (peak.cu): FMAs per second of scalar FFMA and of paired
// FFMA2 (two FMAs each) over the whole device; `sink` holds num_sms * 8 floats.
cudaError_t measure_fp32_peak(int num_sms, float* sink, cudaStream_t s, double* ffma, double* ffma2);


}  // namespace vafr
