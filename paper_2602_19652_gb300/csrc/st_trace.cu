// Ray tracing kernels (Algorithm 1, Sec. III-D filters, Sec. III-E visibility).
//
// Traversal (st_trace_dev.cuh): stack-based walk of the 4-wide BVH (128-byte nodes: the four children's
// boxes as six float4 rows and their references, seven 128-bit loads through the read-only path), the
// nearest hit child next and the others pushed farthest first with their entry distances, skipped on
// pop when a closer hit is known.  Boxes are padded at build time and the slab test widens the far
// distance, so a box is never rejected when the float32 triangle test would hit inside it; the closest
// hit is the smallest (t, triangle index), which makes the result independent of the tree's shape.
//
// Bounces run as a wavefront, one launch per bounce and one more: launch j traces the closest hits of bounce j's live
// rays and, beside them, the visibility rays of bounce j - 1's records (to the receiver reference point, or one per
// microphone), and shades its hits itself (reflection, float64 path length, the record [ray][bounce], the next live
// queue and the next launch's visibility queue).  The kernel is persistent with lane refill: a query advances one wide
// node or one leaf triangle per step, and a lane whose query has finished takes the next one from a warp-aggregated
// atomic counter while the other lanes of its warp continue.  Between the launches of a large call in a two-level scene the
// visibility queue is sorted by hit point.  Results do not depend on the order: closest hits are the smallest (t, triangle
// index), visibility is the absence of any hit in the segment.
// Compiled with -fmad=false (see st_geom.cuh).
#include <algorithm>

#include "st_geom.cuh"
#include "st_internal.cuh"
#include "st_trace_dev.cuh"

namespace st {

namespace {

using namespace trv;

// the traversal view of a scene's arguments (flat, or two-level when `inst` is set)
template <class A>
__host__ __device__ __forceinline__ Trav trav_of(const A& a) {
    Trav T{a.nodes, a.tri_v, a.root, a.max_iter, a.visits, a.stack_limit, a.restarts, a.refill};
    T.bnodes = a.bnodes;
    T.btri = a.btri;
    T.inst = a.inst;
    T.tinst = a.tinst;
    for (int k = 0; k < 6; ++k) T.chk[k] = a.chk[k];
    return T;
}

// traversal kernels: eight 128-thread CTAs per SM (64 registers) on flat scenes, six on two-level ones
// (the object-space ray and the instance state take more registers)
#define ST_TRAV_BOUNDS __launch_bounds__(kTravBlock, TL ? 6 : 8)

// One bounce: closest hits of its live rays (the first bounce: all rays, in direction order), shaded when a lane is
// refilled, and the visibility queries of the bounce before.  Closest hits are claimed first.
// Bound by instruction issue over divergent lanes, and in small calls by the longest query: separate launches for closest
// hits, shading and visibility waited for their slowest query twice a bounce and ran the tail of each alone.  10k rays x
// 3 in the empty room 226 -> 182 us a call, 60k x 4 in light clutter 577 -> 439 us, 100k x 3 in a forest 4726 -> 3598 us,
// 1M x 4 among 1M leaf triangles 15.8 -> 14.6 ms.
template <bool TL>
__global__ void ST_TRAV_BOUNDS k_bounce(const TraceArgs a, int j, int lanes) {
    const Trav T = trav_of(a);
    const int64_t n_closest = j == 0 ? a.N : (j < a.B ? (int64_t)a.n_live[j] : 0);
    const int64_t n_all = n_closest + (j > 0 ? (int64_t)a.n_vis[j - 1] : 0);
    const uint32_t* vis_in = a.vis_q[(j & 1) ^ 1];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int refill = refill_at(T.refill, kRefillClosest, lanes, lanes / 2);
    int2 stack[kStack];
    typename TravStateOf<TL>::type S;
    uint32_t id = 0;  // ray of a closest-hit query, record of a visibility query
    int m = 0;
    bool live = false, hit = false, exhausted = lane >= lanes;
    while (true) {
        if (hit) {  // Algorithm 1's steps after the hit: record, visibility queue, next queue
            hit = false;
            const int32_t tri = S.best;
            const float t = S.tb;
            f3 o, d;
            double r;
            if (j == 0) {
                o = f3{a.s[0], a.s[1], a.s[2]};
                d = rotate(a.q, f3{a.dirs[3 * (size_t)id], a.dirs[3 * (size_t)id + 1], a.dirs[3 * (size_t)id + 2]});
                r = 0.0;
            } else {
                o = f3{a.ox[id], a.oy[id], a.oz[id]};
                d = f3{a.dx[id], a.dy[id], a.dz[id]};
                r = a.racc[id];
            }
            const float tdx = t * d.x, tdy = t * d.y, tdz = t * d.z;
            const f3 P{o.x + tdx, o.y + tdy, o.z + tdz};
            const f3 nv{a.nrm[3 * (size_t)tri], a.nrm[3 * (size_t)tri + 1], a.nrm[3 * (size_t)tri + 2]};
            const float dn = dot(d, nv);
            const float k2 = 2.0f * dn;
            const float knx = k2 * nv.x, kny = k2 * nv.y, knz = k2 * nv.z;
            float len;
            const f3 dr = normalize(f3{d.x - knx, d.y - kny, d.z - knz}, &len);
            r = r + (double)t;
            const size_t rec = (size_t)id * a.B + j;
            a.rec_tri[rec] = tri;
            a.rec_los[rec] = 0;
            a.rec_r[rec] = r;
            a.rec_p[3 * rec] = P.x;
            a.rec_p[3 * rec + 1] = P.y;
            a.rec_p[3 * rec + 2] = P.z;
            a.rec_d[3 * rec] = dr.x;
            a.rec_d[3 * rec + 1] = dr.y;
            a.rec_d[3 * rec + 2] = dr.z;
            // warp-aggregated appends: the record's visibility queries (M with the per-microphone test) ...
            const unsigned active = __activemask();
            const int leader = __ffs(active) - 1, before = __popc(active & ((1u << lane) - 1u));
            const uint32_t per = a.rec_mask ? (uint32_t)a.M : 1u;
            uint32_t base = 0;
            if (lane == leader) base = atomicAdd(a.n_vis + j, (uint32_t)__popc(active) * per);
            base = __shfl_sync(active, base, leader) + (uint32_t)before * per;
            uint32_t* vis_out = a.vis_q[j & 1];
            if (a.rec_mask) {
                a.rec_mask[rec] = 0ull;
                for (uint32_t q = 0; q < per; ++q) vis_out[base + q] = (uint32_t)rec * per + q;
            } else {
                vis_out[base] = (uint32_t)rec;
            }
            if (r < a.r_max && j + 1 < a.B) {  // ... and the live ray
                a.ox[id] = P.x;
                a.oy[id] = P.y;
                a.oz[id] = P.z;
                a.dx[id] = dr.x;
                a.dy[id] = dr.y;
                a.dz[id] = dr.z;
                a.racc[id] = r;
                a.prev[id] = tri;
                const unsigned act = __activemask();
                const int lead = __ffs(act) - 1;
                uint32_t at = 0;
                if (lane == lead) at = atomicAdd(a.n_live + j + 1, (uint32_t)__popc(act));
                at = __shfl_sync(act, at, lead);
                a.live_q[(j + 1) & 1][at + __popc(act & ((1u << lane) - 1u))] = id;
            }
        }
        __syncwarp();
        const bool need = !live && !exhausted;
        const int64_t idx = claim(a.ctr + j, need);
        if (need) {
            if (idx < n_closest) {
                id = j == 0 ? (a.perm ? a.perm[idx] : (uint32_t)idx) : a.live_q[j & 1][idx];
                warp_count(a.queries + 0);
                f3 o, d;
                int32_t prev;
                if (j == 0) {
                    o = f3{a.s[0], a.s[1], a.s[2]};
                    d = rotate(a.q, f3{a.dirs[3 * (size_t)id], a.dirs[3 * (size_t)id + 1], a.dirs[3 * (size_t)id + 2]});
                    prev = -1;
                } else {
                    o = f3{a.ox[id], a.oy[id], a.oz[id]};
                    d = f3{a.dx[id], a.dy[id], a.dz[id]};
                    prev = a.prev[id];
                }
                trav_init(S, T, o, d, prev, a.t_min, __int_as_float(0x7f800000));
                live = true;
            } else if (idx < n_all) {
                id = vis_in[idx - n_closest];
                const float* to = a.R;
                if (a.rec_mask) {  // the entry is record * M + microphone
                    m = (int)(id % (uint32_t)a.M);
                    id /= (uint32_t)a.M;
                    to = a.mics + 3 * m;
                }
                warp_count(a.queries + 1);
                const f3 o{a.rec_p[3 * (size_t)id], a.rec_p[3 * (size_t)id + 1], a.rec_p[3 * (size_t)id + 2]};
                float L;
                const f3 u = normalize(sub(f3{to[0], to[1], to[2]}, o), &L);
                const float tmax = L - a.los_eps;
                if (!(tmax > a.t_min)) {
                    if (a.rec_mask) atomicOr(reinterpret_cast<unsigned long long*>(&a.rec_mask[id]), 1ull << m);
                    a.rec_los[id] = 1;
                } else {
                    trav_init(S, T, o, u, a.rec_tri[id], a.t_min, tmax);
                    S.any = true;
                    live = true;
                }
            } else {
                exhausted = true;
            }
        }
        const unsigned lv0 = __ballot_sync(full, live);
        const unsigned nd0 = __ballot_sync(full, !live && !exhausted);
        if (lv0 == 0u && nd0 == 0u) break;
        while (true) {
            if (live && trav_step<kMixed>(T, S, stack, a.flags)) {
                trav_count_mixed(T, S);
                live = false;
                if (!S.any) {
                    hit = S.best >= 0;
                    ST_CHECK_OR(S.best < a.chk[5], a.flags, hit = false);
                } else if (S.best < 0) {
                    if (a.rec_mask) atomicOr(reinterpret_cast<unsigned long long*>(&a.rec_mask[id]), 1ull << m);
                    a.rec_los[id] = 1;
                }
            }
            const unsigned lv = __ballot_sync(full, live);
            const unsigned nd = __ballot_sync(full, !live && !exhausted);
            if (lv == 0u || __popc(nd) >= refill) break;
        }
    }
}

// Visibility of `target` from the points of a queue (record or candidate ids): out[id] = 1 when no
// triangle other than excl[id] lies on the segment (t_min, |target - p| - eps).
template <bool TL>
__global__ void ST_TRAV_BOUNDS k_visible(const Trav T, const uint32_t* queue, const uint32_t* count,
                                                           const float* pts, const int32_t* excl,
                                                           float tx, float ty, float tz, float t_min, float eps,
                                                           uint8_t* out,
                                                           unsigned long long* ctr, uint32_t* flags,
                                                           unsigned long long* queries, int lanes) {
    const int64_t n = *count;
    const unsigned full = 0xffffffffu;
    const f3 target{tx, ty, tz};
    int2 stack[kStack];
    typename TravStateOf<TL>::type S;
    int64_t id = -1;
    bool live = false, exhausted = (int)(threadIdx.x & 31) >= lanes;
    const int refill = refill_at(T.refill, kRefillAny, lanes, lanes - 4);
    while (true) {
        const bool need = !live && !exhausted;
        const int64_t idx = claim(ctr, need);
        if (need) {
            if (idx < n) {
                id = queue[idx];
                warp_count(queries + 1);
                const f3 o{pts[3 * id], pts[3 * id + 1], pts[3 * id + 2]};
                float L;
                const f3 u = normalize(sub(target, o), &L);
                const float tmax = L - eps;
                if (!(tmax > t_min)) {
                    out[id] = 1;
                } else {
                    trav_init(S, T, o, u, excl[id], t_min, tmax);
                    live = true;
                }
            } else {
                exhausted = true;
            }
        }
        const unsigned lv0 = __ballot_sync(full, live);
        const unsigned nd0 = __ballot_sync(full, !live && !exhausted);
        if (lv0 == 0u && nd0 == 0u) break;
        while (true) {
            if (live && trav_step<kAny>(T, S, stack, flags)) {
                trav_count<true>(T, S);
                out[id] = S.best < 0 ? 1 : 0;
                live = false;
            }
            const unsigned lv = __ballot_sync(full, live);
            const unsigned nd = __ballot_sync(full, !live && !exhausted);
            if (lv == 0u || __popc(nd) >= refill) break;
        }
    }
}

// Sec. III-D: sample g of the global list -> mesh m, local index s; Philox(s, m, pose, 0) selects a
// triangle through the mesh's integer CDF and a barycentric point; then the field-of-view and
// incidence filters; the candidates that pass are queued for the line-of-sight test (k_visible).
__global__ void __launch_bounds__(128, 8) k_diffraction(const DiffArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const f3 s{a.s[0], a.s[1], a.s[2]};
    const f3 fwd{a.fwd[0], a.fwd[1], a.fwd[2]};
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < a.K; g += stride) {
        // mesh: last m with sample_off[m] <= g
        int lo = 0, hi = a.n_obj;  // sample_off has n_obj + 1 entries
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (a.sample_off[mid] <= g) lo = mid; else hi = mid;
        }
        const int m = lo;
        const int64_t sl = g - a.sample_off[m];
        uint32_t x[4];
        philox10((uint32_t)sl, (uint32_t)m, a.pose, 0u, a.seed, x);
        const int64_t b0 = a.mesh_off[m], b1 = a.mesh_off[m + 1];
        const uint64_t W = a.cdf[b1 - 1];
        const uint64_t u = ((uint64_t)x[0] << 32) | x[1];
        const uint64_t target = __umul64hi(u, W);
        int64_t l = b0, h = b1 - 1;
        while (l < h) {
            const int64_t mid = l + ((h - l) >> 1);
            if (a.cdf[mid] > target) h = mid; else l = mid + 1;
        }
        int32_t t = a.mesh_tris[l];
        ST_CHECK_OR(t >= 0 && t < a.chk[5], a.flags, t = 0);
        float ba = (float)(x[2] >> 8) * (1.0f / 16777216.0f);
        float bb = (float)(x[3] >> 8) * (1.0f / 16777216.0f);
        const float sum = ba + bb;
        if (sum > 1.0f) {
            ba = 1.0f - ba;
            bb = 1.0f - bb;
        }
        const float* v0 = a.verts + 3 * (int64_t)a.tris[3 * t];
        const float* v1 = a.verts + 3 * (int64_t)a.tris[3 * t + 1];
        const float* v2 = a.verts + 3 * (int64_t)a.tris[3 * t + 2];
        float p[3];
        for (int k = 0; k < 3; ++k) {
            const float e1 = v1[k] - v0[k];
            const float e2 = v2[k] - v0[k];
            const float p1 = ba * e1;
            const float p2 = bb * e2;
            const float qv = v0[k] + p1;
            p[k] = qv + p2;
        }
        const f3 o{p[0], p[1], p[2]};
        bool ok = true;
        if (a.cos_fov > -1.0f) {
            float L;
            const f3 wn = normalize(sub(o, s), &L);
            if (!(dot(fwd, wn) >= a.cos_fov)) ok = false;
        }
        if (ok) {
            float L;
            const f3 vn = normalize(sub(s, o), &L);
            const f3 n{a.nrm[3 * t], a.nrm[3 * t + 1], a.nrm[3 * t + 2]};
            if (!(fabsf(dot(n, vn)) >= a.cos_inc)) ok = false;
        }
        a.cand_tri[g] = t;
        a.cand_p[3 * g] = p[0];
        a.cand_p[3 * g + 1] = p[1];
        a.cand_p[3 * g + 2] = p[2];
        a.keep[g] = 0;  // set by the line-of-sight kernel for the candidates that passed the filters
        if (ok) {
            const unsigned active = __activemask();
            const int lane = threadIdx.x & 31;
            const int leader = __ffs(active) - 1;
            uint32_t base = 0;
            if (lane == leader) base = atomicAdd(a.los_n, (uint32_t)__popc(active));
            base = __shfl_sync(active, base, leader);
            a.los_q[base + __popc(active & ((1u << lane) - 1u))] = (uint32_t)g;
        }
    }
}

template <bool TL>
__global__ void k_direct(const DirectArgs a) {
    const Trav T = trav_of(a);
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= a.M) return;
    const f3 s{a.s[0], a.s[1], a.s[2]};
    const f3 mic{a.mics[3 * m], a.mics[3 * m + 1], a.mics[3 * m + 2]};
    warp_count(a.queries + 1);
    a.vis[m] = visible<TL>(T, s, mic, -1, a.t_min, a.los_eps, a.flags) ? 1 : 0;
}

// Receiver reference point: float64 sum of the microphones in order, divided by M, rounded.  One thread per
// coordinate adds them in order from shared memory, which all threads fill (one thread doing it all waited for
// each load: 18 us at 64 microphones, before the first visibility ray can start).
constexpr int kCentroidTile = 128;
__global__ void __launch_bounds__(3 * kCentroidTile) k_centroid(const float* mics, int32_t M, float* R) {
    __shared__ float tile[3 * kCentroidTile];
    const int tid = threadIdx.x;
    double acc = 0.0;
    for (int m0 = 0; m0 < M; m0 += kCentroidTile) {
        const int n = min(kCentroidTile, M - m0);
        if (tid < 3 * n) tile[tid] = mics[3 * m0 + tid];
        __syncthreads();
        if (tid < 3)
            for (int m = 0; m < n; ++m) acc += (double)tile[3 * m + tid];
        __syncthreads();
    }
    if (tid < 3) R[tid] = (float)(acc / (double)M);
}

// 10 bits of x spread to every third bit
__device__ __forceinline__ uint32_t spread10(uint32_t x) {
    x &= 0x3ffu;
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

// Morton code (10 bits per axis) of the hit point of every queued visibility query
__global__ void k_vis_keys(const TraceArgs a, int j) {
    const int64_t n = a.n_vis[j];
    const uint32_t* q = a.vis_q[j & 1];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) {
        const float* p = a.rec_p + 3 * (size_t)q[c];
        uint32_t m = 0;
        for (int k = 0; k < 3; ++k) {
            const float u = (p[k] - a.blo[k]) * a.bscale[k];
            m |= spread10((uint32_t)fminf(fmaxf(u, 0.0f), 1023.0f)) << (2 - k);
        }
        a.sort_keys[c] = m;
    }
}

// Morton code (kLosBits per axis) of the candidate point of every queued line-of-sight query
// (line of sight of the clutter workload's 3.2M candidates, sort included: 5 bits 2.42 ms, 8 bits 2.00, 10 bits 1.88)
constexpr int kLosBits = 10;
__global__ void k_los_keys(const DiffArgs a, uint32_t* keys) {
    const int64_t n = *a.los_n;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) {
        const int64_t g = a.los_q[c];
        const float cells = (float)(1 << kLosBits);
        uint32_t m = 0;
        for (int k = 0; k < 3; ++k) {
            const float u = (a.cand_p[3 * g + k] - a.blo[k]) * a.bscale[k] * (cells * (1.0f / 1024.0f));
            m |= spread10((uint32_t)fminf(fmaxf(u, 0.0f), cells - 1.0f)) << (2 - k);
        }
        keys[c] = m;
    }
}

// Octahedral map of a direction to [0,1]^2, 16 bits per axis, Morton-interleaved: nearby directions
// get nearby keys, so sorting by the key groups rays that traverse the same part of the scene.
__device__ __forceinline__ uint32_t spread16(uint32_t x) {
    x &= 0xffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}

// (the lowest bits of the key that the order leaves out: cells of 1/256 of the map's side are below a degree)
constexpr int kDirBits = 16;

__global__ void k_dir_keys(const float* dirs, int64_t n, uint32_t* keys, uint32_t* vals) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        float x = dirs[3 * i], y = dirs[3 * i + 1], z = dirs[3 * i + 2];
        const float l1 = fabsf(x) + fabsf(y) + fabsf(z);
        float px = l1 > 0.0f ? x / l1 : 0.0f, py = l1 > 0.0f ? y / l1 : 0.0f;
        if (z < 0.0f) {
            const float qx = (1.0f - fabsf(py)) * (px >= 0.0f ? 1.0f : -1.0f);
            const float qy = (1.0f - fabsf(px)) * (py >= 0.0f ? 1.0f : -1.0f);
            px = qx;
            py = qy;
        }
        const uint32_t u = (uint32_t)fminf(fmaxf((px + 1.0f) * 32767.5f, 0.0f), 65535.0f);
        const uint32_t v = (uint32_t)fminf(fmaxf((py + 1.0f) * 32767.5f, 0.0f), 65535.0f);
        keys[i] = (spread16(u) << 1) | spread16(v);
        vals[i] = (uint32_t)i;
    }
}

}  // namespace

cudaError_t direction_order(const float* dirs, int64_t n, uint32_t* keys, uint32_t* perm, void* scratch,
                            cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    note_launch();
    k_dir_keys<<<grid_for(n, 256), 256, 0, s>>>(dirs, n, keys, perm);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return radix_sort_u32(keys, perm, n, kDirBits, 32, scratch, s);
}

// Persistent traversal grid for at most n queries: one CTA per resident slot (eight per SM on flat scenes, six on
// two-level ones).  Below one query per lane of that grid the queries are spread over all its warps, a few lanes each
// (at least four): a warp's step then serialises fewer different paths, and the launch ends when its longest query does.
struct TravGrid {
    unsigned ctas;
    int lanes;
};
static TravGrid trav_grid(int64_t n, bool tl, int block = kTravBlock) {
    const int64_t full = 152 * (tl ? 6 : 8) * (kTravBlock / block), warps = full * (block / 32);
    const int lanes = (int)std::min<int64_t>(32, std::max<int64_t>(4, (n + warps - 1) / warps));
    const int64_t per = (int64_t)lanes * (block / 32);
    return TravGrid{(unsigned)std::max<int64_t>(1, std::min<int64_t>(full, (n + per - 1) / per)), lanes};
}

cudaError_t trace_rays(TraceArgs& a, cudaStream_t s, int block) {
    const bool tl = a.inst != nullptr;
    const int threads = std::min(block, kTravBlock);
    for (int j = 0; j <= a.B; ++j) {
        const int64_t most = (j < a.B ? a.N : 0) + (j > 0 ? a.N * (a.rec_mask ? a.M : 1) : 0);
        const TravGrid g = trav_grid(most, tl, threads);
        note_launch();
        if (tl)
            k_bounce<true><<<g.ctas, threads, 0, s>>>(a, j, g.lanes);
        else
            k_bounce<false><<<g.ctas, threads, 0, s>>>(a, j, g.lanes);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (a.sort_keys && j < a.B) {
            note_launch();
            k_vis_keys<<<grid_for(a.N, 256), 256, 0, s>>>(a, j);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if ((e = radix_sort_u32(a.sort_keys, a.vis_q[j & 1], a.N, 0, 30, a.sort_scr, s, a.n_vis + j)) != cudaSuccess)
                return e;
        }
    }
    return cudaSuccess;
}

cudaError_t diffraction_sample(DiffArgs& a, cudaStream_t s) {
    if (a.K <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(a.los_n, 0, sizeof(uint32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(a.ctr, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    note_launch();
    k_diffraction<<<grid_for(a.K, 128, 152 * 16), 128, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (a.sort_keys) {  // stable: equal codes keep the queue order
        note_launch();
        k_los_keys<<<grid_for(a.K, 256), 256, 0, s>>>(a, a.sort_keys);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = radix_sort_u32(a.sort_keys, a.los_q, a.K, 0, 3 * kLosBits, a.sort_scr, s, a.los_n)) != cudaSuccess)
            return e;
    }
    const Trav T = trav_of(a);
    const bool tl = a.inst != nullptr;
    note_launch();
    const TravGrid g = trav_grid(a.K, tl);
    (tl ? k_visible<true> : k_visible<false>)<<<g.ctas, kTravBlock, 0, s>>>(
        T, a.los_q, a.los_n, a.cand_p, a.cand_tri, a.s[0], a.s[1], a.s[2], a.t_min, a.los_eps, a.keep, a.ctr,
        a.flags, a.queries, g.lanes);
    return cudaGetLastError();
}

cudaError_t direct_visibility(DirectArgs& a, cudaStream_t s) {
    if (a.M <= 0) return cudaSuccess;
    note_launch();
    (a.inst ? k_direct<true> : k_direct<false>)<<<(a.M + 63) / 64, 64, 0, s>>>(a);
    return cudaGetLastError();
}

void mic_centroid_host_order(const float* mics_dev, int32_t M, float* R_dev, cudaStream_t s) {
    note_launch();
    k_centroid<<<1, 3 * kCentroidTile, 0, s>>>(mics_dev, M, R_dev);
}

}  // namespace st
