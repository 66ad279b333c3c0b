// pathtrace.cu -- path tracing into the LP buffer and the path-traced
// full-resolution GT (Sec. 8), on the traversal of trace.cuh.
#include "trace.cuh"

namespace vafr {
namespace {

// ---- path tracing into the LP buffer (Sec. 8) ------------------------------------
// The estimator of the ray-casting pipeline's path-traced counterpart: 1 path
// per LP texel, next-event estimation towards the directional light, no Russian
// roulette, at most `depth` diffuse bounces; every surface Lambertian.  Per
// segment: closest hit (ignoring the surface the ray leaves); a miss adds
// beta * sky(d) and ends the path; at a hit (normal n facing the ray, albedo
// rho) the ray origin for what follows is p + 1e-5 max(1, |p|_inf) n; when
// cos = n . (-L) > 0 a shadow ray towards the light (any hit ends it) decides
// whether beta rho cos is added; then, below the depth limit, the next
// direction is cosine-distributed about n (orthonormal basis of Duff et al.
// 2017) and beta *= rho.  Random numbers: the top 24 bits of SplitMix64's
// output function (Steele, Lea, Flood 2014) applied to seed, texel index and
// 2 k + dim in turn.

__device__ __forceinline__ unsigned long long sm64_mix(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ float pt_uniform(unsigned long long seed_h, unsigned long long texel, int k, int dim) {
    const unsigned long long h = sm64_mix(sm64_mix(seed_h ^ texel) ^ (unsigned long long)(2 * k + dim));
    return (float)(h >> 40) * (1.0f / 16777216.0f);
}

__device__ __forceinline__ float3 sky_rgb(float dx, float dy, float dz) {
    const float inv = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    const float s = 0.5f * fmaf(dy, inv, 1.0f);
    return make_float3(1.0f - 0.5f * s, 1.0f - 0.3f * s, 1.0f);
}

// Unit geometric normal of the hit leaf, turned to face the ray.
__device__ __forceinline__ float3 face_normal(const SceneDev& sc, const Ray& r, int leaf) {
    const float4 a = __ldg(sc.leaves + 3ll * leaf);
    const float4 b = __ldg(sc.leaves + 3ll * leaf + 1);
    const float4 c = __ldg(sc.leaves + 3ll * leaf + 2);
    const float e1x = b.x - a.x, e1y = b.y - a.y, e1z = b.z - a.z;
    const float e2x = c.x - a.x, e2y = c.y - a.y, e2z = c.z - a.z;
    float nx = e1y * e2z - e1z * e2y;
    float ny = e1z * e2x - e1x * e2z;
    float nz = e1x * e2y - e1y * e2x;
    const float inv = rsqrtf(fmaf(nx, nx, fmaf(ny, ny, nz * nz)));
    nx *= inv; ny *= inv; nz *= inv;
    if (fmaf(nx, r.dx, fmaf(ny, r.dy, nz * r.dz)) > 0.0f) { nx = -nx; ny = -ny; nz = -nz; }
    return make_float3(nx, ny, nz);
}

// A warp keeps a pool of paths, one record per path that still has a ray to
// trace: a closest-hit segment or a shadow ray.  It traces 32 records at a
// time, whatever their depth and kind, and returns the paths that go on to the
// pool; whenever fewer than 32 are left it starts the next 32 paths.  So every
// traversal has 32 rays until the work runs out, and the primary rays of a
// chunk are still traced together.
//
// One path per lane from its first to its last segment leaves most lanes idle:
// on the 1.07 M triangle terrain 93 % of the paths have a second segment but
// 25 % a third and 16 % a fourth, and 14 %, 12 % and 7 % a shadow ray there,
// while each of these steps takes a warp nearly as long as the full ones (276,
// 629, 974 and 1,252 us for the LP buffer at 0 to 3 bounces, 10.6 of 32 lanes
// active).  With the pool 1,252 us become 945 (15 lanes; the incoherent bounce
// rays' leaf tests and pushes are what diverges now).
// The records also hold what the traversal does not need, so it fits 64
// registers and kPathBlocks blocks per SM (one path per lane: 93 and 5).  When
// the pool was made, on a traversal of more instructions that took 1,391 us with one
// path per lane, 6, 7 and 8 blocks measured 1,156, 1,148 and 1,110 us, and 1,064
// with all four children sorted.  What a ray does not need lies in global memory
// instead of beside it in shared memory, where it took L1 from the nodes (1,172
// us then).
constexpr int kPathBlocks = 8;   // resident blocks per SM that the launch and its scratch count on
constexpr int kPoolPaths = 64;   // fewer than 32 waiting, and the next 32
struct PathPool {
    float o[3][kPoolPaths], d[3][kPoolPaths];   // next ray's origin; direction of the next closest-hit segment
    int skip[kPoolPaths];                       // triangle the ray leaves
    unsigned work[kPoolPaths];                  // work item (texel or pixel)
    unsigned step[kPoolPaths];                  // 2 x segment, + 1: its shadow ray
};
// The rest of a record, in global memory (L2): read and written once per ray,
// and not before a path's first hit (until then beta is 1, the rest 0).
struct PathState {
    float beta[3][kPoolPaths], acc[3][kPoolPaths];
    float cosl[kPoolPaths];      // shadow ray: cosine towards the light
    unsigned mask[kPoolPaths];   // signature: shadow rays lit / cast
};

// LP texel (slot and the guard slots that copy it) or display pixel of a work
// item, and its random-number key.
struct PathPlace {
    int slot, glo, ghi;
    long long px;
    unsigned long long key;
};

// Display pixel (x, y) of GT work item `local`; false when outside the display.
__device__ __forceinline__ bool gt_pixel(const FrameDesc& f, long long local, int& x, int& y) {
    const long long tile = local >> 5;
    const int in = (int)(local & 31);
    const int tiles_x = (f.W + 7) >> 3;
    x = (int)(tile % tiles_x) * 8 + (in & 7);
    y = (int)(tile / tiles_x) * 4 + (in >> 3);
    return x < f.W && y < f.H;
}

template <bool GT>
__device__ __forceinline__ PathPlace path_place(const FrameDesc& f, long long local) {
    PathPlace p{0, -1, -1, 0, 0ull};
    if (GT) {
        int x, y;
        gt_pixel(f, local, x, y);
        p.px = (long long)y * f.W + x;
        p.key = (unsigned long long)p.px;
    } else {
        const int2 tc = __ldg(f.work + local);
        const int2 cc = __ldg(&f.col[tc.y]);
        p.slot = tc.x;
        p.glo = tc.x - cc.x == cc.y - 1 ? tc.x - cc.y : -1;
        p.ghi = tc.x == cc.x ? tc.x + cc.y : -1;
        p.key = (unsigned long long)(tc.x - (2 * tc.y + 1));   // index in column order, no guards
    }
    return p;
}

// Primary ray of a work item; false when it is outside the display.
template <bool GT>
__device__ __forceinline__ bool path_ray(const FrameDesc& f, long long local, Ray& r) {
    if (!GT) {
        int glo, ghi;
        lp_ray(f, (int)local, r, glo, ghi);
        return true;
    }
    int x, y;
    if (!gt_pixel(f, local, x, y)) return false;
    world_ray(f, f.cr * ((float)x + 0.5f - 0.5f * (float)f.W), f.cr * (0.5f * (float)f.H - ((float)y + 0.5f)), r);
    return true;
}

template <bool GT>
__device__ __forceinline__ void store_path(const FrameDesc& f, const PathPlace& p, float4 v) {
    if (GT) {
        store_px(f.disp, p.px, f.disp_fmt, v);
    } else {
        store_px(f.lp, p.slot, f.lp_fmt, v);
        if (p.glo >= 0) store_px(f.lp, p.glo, f.lp_fmt, v);
        if (p.ghi >= 0) store_px(f.lp, p.ghi, f.lp_fmt, v);
    }
}

// Surface point of hit h of ray r, off the surface along the facing normal n.
__device__ __forceinline__ void leave_surface(const Ray& r, const Hit& h, const float3& n, float o[3]) {
    const float px = fmaf(h.t, r.dx, r.ox), py = fmaf(h.t, r.dy, r.oy), pz = fmaf(h.t, r.dz, r.oz);
    const float off = 1e-5f * fmaxf(1.0f, fmaxf(fabsf(px), fmaxf(fabsf(py), fabsf(pz))));
    o[0] = fmaf(off, n.x, px);
    o[1] = fmaf(off, n.y, py);
    o[2] = fmaf(off, n.z, pz);
}

// Direction of the next segment: cosine-distributed about n.
__device__ __forceinline__ void bounce(const float3& nn, unsigned long long seed_h, unsigned long long key, int k,
                                       float d[3]) {
    const float u1 = pt_uniform(seed_h, key, k, 0), u2 = pt_uniform(seed_h, key, k, 1);
    float sp, cp;
    sincospif(2.0f * u2, &sp, &cp);
    const float rr = sqrtf(u1);
    const float lx = rr * cp, ly = rr * sp, lz = sqrtf(fmaxf(0.0f, 1.0f - u1));
    const float sg = copysignf(1.0f, nn.z);
    const float aa = -1.0f / (sg + nn.z);
    const float bb = nn.x * nn.y * aa;
    const float t1x = 1.0f + sg * nn.x * nn.x * aa, t1y = sg * bb, t1z = -sg * nn.x;
    const float t2x = bb, t2y = sg + nn.y * nn.y * aa, t2z = -nn.y;
    d[0] = fmaf(lx, t1x, fmaf(ly, t2x, lz * nn.x));
    d[1] = fmaf(lx, t1y, fmaf(ly, t2y, lz * nn.y));
    d[2] = fmaf(lx, t1z, fmaf(ly, t2z, lz * nn.z));
}

// Path signature (LP only): depth + 2 ints per slot: hit id per segment, -1
// miss, -2 not traced; then the shadow mask: bit k = segment k's shadow ray
// reached the light, bit 16 + k = it was cast.
//
// One path per lane from its first to its last segment: the choice for little
// work (launch_path_one).
template <int TPB, int ORDER, bool GT, class B>
__global__ void __launch_bounds__(TPB)
k_path_lanes(const SceneDev sc, const __grid_constant__ B b, unsigned long long seed, int depth) {
    const int lane = threadIdx.x & 31;
    const unsigned long long seed_h = sm64_mix(seed);
    const float tlx = -sc.light[0], tly = -sc.light[1], tlz = -sc.light[2];
    while (true) {
        unsigned long long base = 0ull;
        if (lane == 0) base = atomicAdd(b.work_counter, 32ull);
        base = __shfl_sync(0xffffffffu, base, 0);
        if ((long long)base >= b.total_work) break;
        const long long w = (long long)base + lane;
        if (w >= b.total_work) continue;
        const FrameDesc& f = b.d[find_frame(b, w, false)];
        Ray r;
        if (!path_ray<GT>(f, w - f.work_begin, r)) continue;
        const PathPlace at = path_place<GT>(f, w - f.work_begin);
        int* sig = !GT && f.hit_ids ? f.hit_ids + (long long)at.slot * (depth + 2) : nullptr;
        float beta[3] = {1.0f, 1.0f, 1.0f}, acc[3] = {0.0f, 0.0f, 0.0f};
        unsigned mask = 0u, fault = 0u;
        int k = 0;
        for (; k <= depth; ++k) {
            ray_setup(r);
            Hit h;
            fault |= traverse4<false, ORDER, true>(sc, r, h, nullptr, nullptr, nullptr);
            if (sig) sig[k] = h.leaf >= 0 ? h.id : -1;
            if (h.leaf < 0) {
                const float3 sky = sky_rgb(r.dx, r.dy, r.dz);
                acc[0] = fmaf(beta[0], sky.x, acc[0]);
                acc[1] = fmaf(beta[1], sky.y, acc[1]);
                acc[2] = fmaf(beta[2], sky.z, acc[2]);
                ++k;
                break;
            }
            const float3 n = face_normal(sc, r, h.leaf);
            float o[3];
            leave_surface(r, h, n, o);
            const float4 rho = __ldg(sc.albedo + h.id);
            beta[0] *= rho.x; beta[1] *= rho.y; beta[2] *= rho.z;
            const float cosl = fmaf(n.x, tlx, fmaf(n.y, tly, n.z * tlz));
            r.ox = o[0]; r.oy = o[1]; r.oz = o[2];
            r.skip = h.id;
            if (cosl > 0.0f) {   // a shadow ray is cast
                mask |= 1u << (16 + k);
                r.dx = tlx; r.dy = tly; r.dz = tlz;
                ray_setup(r);
                Hit hs;
                fault |= traverse4<false, ORDER, true>(sc, r, hs, nullptr, nullptr, nullptr, true);
                if (hs.leaf < 0) {
                    mask |= 1u << k;
#pragma unroll
                    for (int c = 0; c < 3; ++c) acc[c] = fmaf(beta[c], cosl, acc[c]);
                }
            }
            if (k < depth) {
                float d[3];
                bounce(n, seed_h, at.key, k, d);
                r.dx = d[0]; r.dy = d[1]; r.dz = d[2];
            }
        }
        if (fault) atomicOr(f.status, fault);
        store_path<GT>(f, at, make_float4(acc[0], acc[1], acc[2], 1.0f));
        if (sig) {
            for (k = min(k, depth + 1); k <= depth; ++k) sig[k] = -2;
            sig[depth + 1] = (int)mask;
        }
    }
}

template <int TPB, int ORDER, bool GT, int MINB, class B>
__global__ void __launch_bounds__(TPB, MINB)
k_path(const SceneDev sc, const __grid_constant__ B b, unsigned long long seed, int depth, PathState* states) {
    __shared__ PathPool pools[TPB / 32];
    PathPool& P = pools[threadIdx.x >> 5];
    PathState& S = states[blockIdx.x * (TPB / 32) + (threadIdx.x >> 5)];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned long long seed_h = sm64_mix(seed);
    const float tlx = -sc.light[0], tly = -sc.light[1], tlz = -sc.light[2];
    int count = 0;          // records in the pool
    bool more = true;       // work items left
    while (true) {
        if (count < 32 && more) {   // the next 32 paths
            unsigned long long base = 0ull;
            if (lane == 0) base = atomicAdd(b.work_counter, 32ull);
            base = __shfl_sync(full, base, 0);
            more = (long long)base < b.total_work;
            const long long w = (long long)base + lane;
            Ray r;
            bool live = w < b.total_work;
            if (live) {
                const FrameDesc& f = b.d[find_frame(b, w, false)];
                live = path_ray<GT>(f, w - f.work_begin, r);
            }
            const unsigned lm = __ballot_sync(full, live);
            if (live) {
                const int q = count + __popc(lm & ((1u << lane) - 1u));
                P.o[0][q] = r.ox; P.o[1][q] = r.oy; P.o[2][q] = r.oz;
                P.d[0][q] = r.dx; P.d[1][q] = r.dy; P.d[2][q] = r.dz;
                P.skip[q] = -1;
                P.work[q] = (unsigned)w;
                P.step[q] = 0u;
            }
            count += __popc(lm);
            __syncwarp();
            if (count < 32 && more) continue;
        }
        if (count == 0) break;
        // Once the work has run out and 16 records or fewer are left, a record at
        // a shadow ray also gets its next segment traced, by lane + 16: the paths
        // that end the launch take fewer steps.
        const bool pairs = !more && count <= 16;
        const int n = min(count, 32);
        const int idx = pairs ? lane & 15 : lane;
        const bool second = pairs && lane >= 16;
        const int q = count - n + idx;   // this lane's record
        const bool on = idx < n && !second;
        Hit h;
        h.t = INFINITY;
        h.leaf = -1;
        h.id = INT_MAX;
        if (on || (second && idx < n && (P.step[q] & 1u) && (int)(P.step[q] >> 1) < depth)) {
            const bool shadow = on && (P.step[q] & 1u);
            Ray r;
            r.ox = P.o[0][q]; r.oy = P.o[1][q]; r.oz = P.o[2][q];
            r.dx = shadow ? tlx : P.d[0][q];
            r.dy = shadow ? tly : P.d[1][q];
            r.dz = shadow ? tlz : P.d[2][q];
            r.skip = P.skip[q];
            ray_setup(r);
            const unsigned fault = traverse4<false, ORDER, true>(sc, r, h, nullptr, nullptr, nullptr, shadow);
            if (fault) atomicOr(b.d[find_frame(b, (long long)P.work[q], false)].status, fault);
        }
        __syncwarp();
        Hit next = h;      // closest hit of this lane's record, where it was traced
        if (pairs) {
            const int src = idx + 16;
            const float t2 = __shfl_sync(full, h.t, src);
            const int leaf2 = __shfl_sync(full, h.leaf, src), id2 = __shfl_sync(full, h.id, src);
            if (on && (P.step[q] & 1u)) {
                next.t = t2;
                next.leaf = leaf2;
                next.id = id2;
            }
        }
        bool go = false;   // the path has another ray
        float o[3], d[3], beta[3] = {1.0f, 1.0f, 1.0f}, acc[3] = {0.0f, 0.0f, 0.0f}, cosl = 0.0f;
        int skip = -1;
        unsigned work = 0u, step = 0u, mask = 0u;
        if (on) {
            work = P.work[q];
            step = P.step[q];
            skip = P.skip[q];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                o[c] = P.o[c][q];
                d[c] = P.d[c][q];
            }
            if (step) {
                mask = __ldcg(&S.mask[q]);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    beta[c] = __ldcg(&S.beta[c][q]);
                    acc[c] = __ldcg(&S.acc[c][q]);
                }
            }
            int k = (int)(step >> 1);
            const FrameDesc& f = b.d[find_frame(b, (long long)work, false)];
            const PathPlace at = path_place<GT>(f, (long long)work - f.work_begin);
            int* sig = !GT && f.hit_ids ? f.hit_ids + (long long)at.slot * (depth + 2) : nullptr;
            bool closest = !(step & 1u);
            if (!closest) {
                if (h.leaf < 0) {
                    cosl = __ldcg(&S.cosl[q]);
                    mask |= 1u << k;
#pragma unroll
                    for (int c = 0; c < 3; ++c) acc[c] = fmaf(beta[c], cosl, acc[c]);
                }
                if (k < depth) {
                    go = true;
                    step = 2u * (unsigned)++k;
                    closest = pairs;
                }
            }
            if (closest) {
                go = false;
                if (sig) sig[k] = next.leaf >= 0 ? next.id : -1;
                if (next.leaf < 0) {
                    const float3 sky = sky_rgb(d[0], d[1], d[2]);
                    acc[0] = fmaf(beta[0], sky.x, acc[0]);
                    acc[1] = fmaf(beta[1], sky.y, acc[1]);
                    acc[2] = fmaf(beta[2], sky.z, acc[2]);
                } else {
                    Ray r;
                    r.ox = o[0]; r.oy = o[1]; r.oz = o[2];
                    r.dx = d[0]; r.dy = d[1]; r.dz = d[2];
                    const float3 nn = face_normal(sc, r, next.leaf);
                    leave_surface(r, next, nn, o);
                    const float4 rho = __ldg(sc.albedo + next.id);
                    beta[0] *= rho.x; beta[1] *= rho.y; beta[2] *= rho.z;
                    skip = next.id;
                    cosl = fmaf(nn.x, tlx, fmaf(nn.y, tly, nn.z * tlz));
                    if (k < depth) {
                        bounce(nn, seed_h, at.key, k, d);
                    }
                    if (cosl > 0.0f) {   // a shadow ray is cast
                        mask |= 1u << (16 + k);
                        step += 1u;
                        go = true;
                    } else {
                        step += 2u;
                        go = k < depth;
                    }
                }
            }
            if (!go) {
                store_path<GT>(f, at, make_float4(acc[0], acc[1], acc[2], 1.0f));
                if (sig) {
                    for (int j = k + 1; j <= depth; ++j) sig[j] = -2;
                    sig[depth + 1] = (int)mask;
                }
            }
        }
        __syncwarp();
        const unsigned gm = __ballot_sync(full, go);
        count -= n;
        if (go) {
            const int z = count + __popc(gm & ((1u << lane) - 1u));
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                P.o[c][z] = o[c];
                P.d[c][z] = d[c];
                __stcg(&S.beta[c][z], beta[c]);
                __stcg(&S.acc[c][z], acc[c]);
            }
            __stcg(&S.cosl[z], cosl);
            __stcg(&S.mask[z], mask);
            P.skip[z] = skip;
            P.work[z] = work;
            P.step[z] = step;
        }
        count += __popc(gm);
        __syncwarp();
    }
}

template <bool GT, class B>
cudaError_t launch_path_one(const SceneDev& sc, const B& b, unsigned long long seed, int depth, void* scratch,
                            cudaStream_t s, int num_sms) {
    if (b.total_work <= 0) return cudaSuccess;
    constexpr int TPB = 128;
    auto pooled = k_path<TPB, 0, GT, kPathBlocks, B>;
    auto lanes = k_path_lanes<TPB, 1, GT, B>;
    const bool pool = scratch != nullptr;
    int per_sm = 0;
    cudaError_t e = pool ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pooled, TPB, 0)
                         : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lanes, TPB, 0);
    if (e != cudaSuccess) return e;
    per_sm = min(max(per_sm, 1), kPathBlocks);   // the scratch holds this many blocks' pools
    e = cudaMemsetAsync(b.work_counter, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    long long grid = (long long)per_sm * num_sms;
    const long long need = (b.total_work + TPB - 1) / TPB;
    if (need < grid) grid = need < 1 ? 1 : need;
    if (pool)
        pooled<<<(unsigned)grid, TPB, 0, s>>>(sc, b, seed, depth, static_cast<PathState*>(scratch));
    else
        lanes<<<(unsigned)grid, TPB, 0, s>>>(sc, b, seed, depth);
    count_launch(1);
    return cudaGetLastError();
}
}  // namespace

// Gathering the paths pays once enough of them go on: the pool's last paths of
// each warp take a step at a time with few lanes, some tenths of a launch of
// one LP buffer.  Measured at 0.7 and 1.06 M texels on terrains of 7 K to 1.07 M
// triangles, one path per lane against the pool: no bounce 150 against 158 us
// (the shadow rays keep nine lanes in ten busy anyway), one bounce 287 against
// 288 and 142 against 146, two 283 against 286 (0.7 M) and 411 against 399
// (1.06 M), three 352 against 364 (0.7 M) and 528 against 497 (1.06 M); two at
// 2.07 M pixels 1,440 against 1,139.  So the line lies at 2.5 M bounces.
bool path_uses_pool(long long work, int depth) { return (long long)depth * work >= 2500000; }

size_t path_scratch_bytes(int num_sms) {
    return sizeof(PathState) * (size_t)num_sms * kPathBlocks * 4;
}

template <class B>
cudaError_t launch_path_lp(const SceneDev& scene, const B& batch, unsigned long long seed, int depth,
                           void* scratch, cudaStream_t s, int num_sms) {
    return launch_path_one<false>(scene, batch, seed, depth, scratch, s, num_sms);
}
template <class B>
cudaError_t launch_path_gt(const SceneDev& scene, const B& batch, unsigned long long seed, int depth,
                           void* scratch, cudaStream_t s, int num_sms) {
    return launch_path_one<true>(scene, batch, seed, depth, scratch, s, num_sms);
}
template cudaError_t launch_path_gt<SmallBatch>(const SceneDev&, const SmallBatch&, unsigned long long, int, void*,
                                                cudaStream_t, int);
template cudaError_t launch_path_lp<SmallBatch>(const SceneDev&, const SmallBatch&, unsigned long long, int, void*,
                                                cudaStream_t, int);
template cudaError_t launch_path_lp<BigBatch>(const SceneDev&, const BigBatch&, unsigned long long, int, void*,
                                              cudaStream_t, int);

}  // namespace vafr
