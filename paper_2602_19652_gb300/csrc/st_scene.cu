// Scene pre-processing on the device (Sec. III-B, Sec. III-D):
//   validation, geometric normals, vertex welding, one-ring adjacency (ascending triangle ids),
//   Meyer mean curvature G_v, the triangle metric C_i (Eq. 1), per-mesh dithered integer CDFs and
//   diffraction sample counts, and a BVH (Morton codes, radix sort, clusters merged by least surface,
//   bottom-up boxes, small subtrees collapsed into leaves of <= 4 triangles).
// Compiled with -fmad=false: curvature and CDF weights decide which triangles are sampled.
#include <math.h>

#include <algorithm>
#include <cstring>
#include <string>

#include "st_geom.cuh"
#include "st_internal.cuh"

namespace st {

namespace {

#define CK(x)                                \
    do {                                     \
        cudaError_t e_ = (x);                \
        if (e_ != cudaSuccess) return e_;    \
    } while (0)

constexpr int kB = 256;

__device__ __forceinline__ f3 vload(const float* V, int64_t i) { return f3{V[3 * i], V[3 * i + 1], V[3 * i + 2]}; }

__global__ void k_validate(const float* V, int64_t nv, const int32_t* T, int64_t nt, const int32_t* mat,
                           int32_t n_mat, const int32_t* obj, uint32_t* flags) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv + nt; i += stride) {
        if (i < nv) {
            float x = V[3 * i], y = V[3 * i + 1], z = V[3 * i + 2];
            if (!(isfinite(x) && isfinite(y) && isfinite(z))) atomicOr(flags, kFlagBadVertex);
        } else {
            int64_t t = i - nv;
            for (int k = 0; k < 3; ++k) {
                int32_t v = T[3 * t + k];
                if (v < 0 || v >= nv) atomicOr(flags, kFlagBadIndex);
            }
            if (mat[t] < 0 || mat[t] >= n_mat || obj[t] < 0) atomicOr(flags, kFlagBadIndex);
        }
    }
}

__global__ void k_normals(const float* V, const int32_t* T, int64_t nt, float* N) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride) {
        f3 a = vload(V, T[3 * t]), b = vload(V, T[3 * t + 1]), c = vload(V, T[3 * t + 2]);
        float l;
        f3 n = normalize(cross(sub(b, a), sub(c, a)), &l);
        N[3 * t] = n.x;
        N[3 * t + 1] = n.y;
        N[3 * t + 2] = n.z;
    }
}

// ---------------------------------------------------------------- welding
__device__ __forceinline__ uint32_t pos_bits(float x) { return __float_as_uint(x + 0.0f); }  // -0 -> +0

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z ^= z >> 33;
    z *= 0xff51afd7ed558ccdull;
    z ^= z >> 33;
    z *= 0xc4ceb9fe1a85ec53ull;
    z ^= z >> 33;
    return z;
}

// (32 bits of the hash: equal positions get equal keys, and k_weld_runs compares the positions of a run anyway)
__global__ void k_pos_keys(const float* V, int64_t nv, uint32_t* keys, uint32_t* vals) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += stride) {
        uint64_t h = mix64(pos_bits(V[3 * i]));
        h = mix64(h ^ pos_bits(V[3 * i + 1]));
        h = mix64(h ^ ((uint64_t)pos_bits(V[3 * i + 2]) << 17));
        keys[i] = (uint32_t)(h >> 32);
        vals[i] = (uint32_t)i;
    }
}

__device__ __forceinline__ bool same_pos(const float* V, uint32_t a, uint32_t b) {
    return pos_bits(V[3 * (int64_t)a]) == pos_bits(V[3 * (int64_t)b]) &&
           pos_bits(V[3 * (int64_t)a + 1]) == pos_bits(V[3 * (int64_t)b + 1]) &&
           pos_bits(V[3 * (int64_t)a + 2]) == pos_bits(V[3 * (int64_t)b + 2]);
}

// One thread per run of equal hashes: canon[v] = smallest index with exactly the same position.
__global__ void k_weld_runs(const float* V, int64_t nv, const uint32_t* keys, const uint32_t* vals, int32_t* canon) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += stride) {
        if (i > 0 && keys[i] == keys[i - 1]) continue;
        int64_t j = i + 1;
        while (j < nv && keys[j] == keys[i]) ++j;
        for (int64_t a = i; a < j; ++a) {
            uint32_t va = vals[a];
            uint32_t best = va;
            for (int64_t b = i; b < j; ++b) {
                uint32_t vb = vals[b];
                if (vb < best && same_pos(V, va, vb)) best = vb;
            }
            canon[va] = (int32_t)best;
        }
    }
}

// ---------------------------------------------------------------- adjacency
__device__ __forceinline__ bool tri_corner_dup(const int32_t* canon, const int32_t* T, int64_t t, int k) {
    int32_t c = canon[T[3 * t + k]];
    for (int q = 0; q < k; ++q)
        if (canon[T[3 * t + q]] == c) return true;
    return false;
}

__global__ void k_adj_count(const int32_t* canon, const int32_t* T, int64_t nt, uint32_t* cnt) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride)
        for (int k = 0; k < 3; ++k)
            if (!tri_corner_dup(canon, T, t, k)) atomicAdd(&cnt[canon[T[3 * t + k]]], 1u);
}

__global__ void k_adj_fill(const int32_t* canon, const int32_t* T, int64_t nt, const uint32_t* off, uint32_t* cursor,
                           int32_t* adj) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride)
        for (int k = 0; k < 3; ++k)
            if (!tri_corner_dup(canon, T, t, k)) {
                int32_t c = canon[T[3 * t + k]];
                uint32_t p = atomicAdd(&cursor[c], 1u);
                adj[off[c] + p] = (int32_t)t;
            }
}

__global__ void k_adj_sort(int64_t nv, const uint32_t* off, int32_t* adj) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += stride) {
        uint32_t a = off[v], b = off[v + 1];
        for (uint32_t i = a + 1; i < b; ++i) {
            int32_t x = adj[i];
            uint32_t j = i;
            while (j > a && adj[j - 1] > x) {
                adj[j] = adj[j - 1];
                --j;
            }
            adj[j] = x;
        }
    }
}

// ---------------------------------------------------------------- Meyer curvature (Sec. III-B)
// For canonical vertex v and each incident triangle (v, a, b) in ascending triangle index:
//   cot at a = (v-a).(b-a) / |(a-v) x (b-v)|, cot at b = (v-b).(a-b) / |(a-v) x (b-v)|,
//   sum += cot_b (v - a) + cot_a (v - b); A_mixed += Voronoi area, or area/2 (obtuse at v),
//   or area/4 (obtuse elsewhere);  G_v = |sum / (2 A_mixed)| / 2.
__global__ void k_curvature(const float* V, int64_t nv, const int32_t* T, const int32_t* canon, const uint32_t* off,
                            const int32_t* adj, float* Gc) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += stride) {
        if (canon[v] != v) continue;
        f3 xv = vload(V, v);
        float Sx = 0.0f, Sy = 0.0f, Sz = 0.0f, Amix = 0.0f;
        for (uint32_t e = off[v]; e < off[v + 1]; ++e) {
            int64_t t = adj[e];
            int32_t c0 = canon[T[3 * t]], c1 = canon[T[3 * t + 1]], c2 = canon[T[3 * t + 2]];
            if (c0 == c1 || c1 == c2 || c0 == c2) continue;
            int32_t ia, ib;
            if (c0 == v) {
                ia = c1;
                ib = c2;
            } else if (c1 == v) {
                ia = c2;
                ib = c0;
            } else {
                ia = c0;
                ib = c1;
            }
            f3 xa = vload(V, ia), xb = vload(V, ib);
            f3 va = sub(xv, xa), ba = sub(xb, xa), vb = sub(xv, xb), ab = sub(xa, xb), av = sub(xa, xv),
               bv = sub(xb, xv);
            f3 cr = cross(av, bv);
            float cross_len = sqrtf(dot(cr, cr));
            if (!(cross_len > 0.0f)) continue;
            float cot_a = dot(va, ba) / cross_len;
            float cot_b = dot(vb, ab) / cross_len;
            {
                float t1 = cot_b * va.x, t2 = cot_a * vb.x;
                Sx = Sx + (t1 + t2);
                t1 = cot_b * va.y;
                t2 = cot_a * vb.y;
                Sy = Sy + (t1 + t2);
                t1 = cot_b * va.z;
                t2 = cot_a * vb.z;
                Sz = Sz + (t1 + t2);
            }
            float area = 0.5f * cross_len;
            float dv = dot(av, bv), da = dot(va, ba), db = dot(vb, ab);
            float amix;
            if (dv < 0.0f)
                amix = area / 2.0f;
            else if (da < 0.0f || db < 0.0f)
                amix = area / 4.0f;
            else {
                float lvb = dot(vb, vb), lva = dot(va, va);
                float p1 = lvb * cot_a, p2 = lva * cot_b;
                amix = (p1 + p2) / 8.0f;
            }
            Amix = Amix + amix;
        }
        float g = 0.0f;
        if (Amix > 0.0f) {
            float den = 2.0f * Amix;
            f3 K{Sx / den, Sy / den, Sz / den};
            g = 0.5f * sqrtf(dot(K, K));
        }
        Gc[v] = g;
    }
}

__global__ void k_expand_G(const int32_t* canon, int64_t nv, const float* Gc, float* G) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += stride) G[v] = Gc[canon[v]];
}

// Eq. 1: C_i = eta * w(A_i) * (max G - min G), w(A) = clamp(A / A_ref, 0, 1).
__global__ void k_metric(const float* V, const int32_t* T, int64_t nt, const int32_t* canon, const float* G, float eta,
                         float area_ref, float* C, uint32_t* cmax_bits, const int32_t* obj) {
    const int lane = threadIdx.x & 31;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < nt; t0 += stride) {
        const int64_t t = t0 + lane;
        int32_t m = -1;
        float c = 0.0f;
        if (t < nt) {
            m = obj[t];
            int32_t i0 = T[3 * t], i1 = T[3 * t + 1], i2 = T[3 * t + 2];
            if (!(canon[i0] == canon[i1] || canon[i1] == canon[i2] || canon[i0] == canon[i2])) {
                f3 a = vload(V, i0);
                f3 cr = cross(sub(vload(V, i1), a), sub(vload(V, i2), a));
                float A = 0.5f * sqrtf(dot(cr, cr));
                if (A > 0.0f) {
                    float w = A / area_ref;
                    if (w > 1.0f) w = 1.0f;
                    if (w < 0.0f) w = 0.0f;
                    float g0 = G[i0], g1 = G[i1], g2 = G[i2];
                    float gmax = fmaxf(fmaxf(g0, g1), g2), gmin = fminf(fminf(g0, g1), g2);
                    float ew = eta * w;
                    c = ew * (gmax - gmin);
                }
            }
            C[t] = c;
        }
        const uint32_t same = __match_any_sync(0xffffffffu, m);
        const uint32_t top = __reduce_max_sync(same, __float_as_uint(c));  // c >= 0: bit order = value order
        if (m >= 0 && lane == __ffs(same) - 1) atomicMax(&cmax_bits[m], top);
    }
}

// ---------------------------------------------------------------- diffraction CDFs (Sec. III-D)
__device__ __forceinline__ void philox10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint64_t seed,
                                         uint32_t out[4]) {
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        if (round > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
        uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
        uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
    }
    out[0] = c0;
    out[1] = c1;
    out[2] = c2;
    out[3] = c3;
}

__global__ void k_widen(const uint32_t* in, int64_t n, int64_t* out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = in[i];
}
__global__ void k_mesh_count(const int32_t* obj, int64_t nt, uint32_t* cnt) {
    const int lane = threadIdx.x & 31;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; t0 < nt; t0 += stride) {
        const int32_t m = t0 + lane < nt ? obj[t0 + lane] : -1;
        const uint32_t same = __match_any_sync(0xffffffffu, m);
        if (m >= 0 && lane == __ffs(same) - 1) atomicAdd(&cnt[m], (uint32_t)__popc(same));
    }
}

__global__ void k_mesh_keys(const int32_t* obj, int64_t nt, uint32_t* keys, uint32_t* vals) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride) {
        keys[t] = (uint32_t)obj[t];
        vals[t] = (uint32_t)t;
    }
}

__global__ void k_quantize(const int32_t* mesh_tris, int64_t nt, const int32_t* obj, const float* C,
                           const uint32_t* cmax_bits, uint64_t* Q, unsigned long long* sumQ) {
    const int lane = threadIdx.x & 31;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; i0 < nt; i0 += stride) {
        const int64_t i = i0 + lane;
        int32_t m = -1;
        uint64_t q = 0;  // at most 2^24, unless the metric is not finite
        if (i < nt) {
            const int32_t t = mesh_tris[i];
            m = obj[t];
            const float cmax = __uint_as_float(cmax_bits[m]);
            if (cmax > 0.0f) {
                float r = C[t] / cmax;
                float s = r * 16777216.0f;
                q = (uint64_t)floorf(s);
            }
            Q[i] = q;
        }
        const uint32_t same = __match_any_sync(0xffffffffu, m);
        const uint32_t sum = __reduce_add_sync(same, q <= 16777216u ? (uint32_t)q : 0u);
        if (q > 16777216u) atomicAdd(&sumQ[m], (unsigned long long)q);
        if (m >= 0 && lane == __ffs(same) - 1) atomicAdd(&sumQ[m], (unsigned long long)sum);
    }
}

__global__ void k_dither(const int32_t* mesh_tris, int64_t nt, const int32_t* obj, const uint32_t* mesh_off,
                         const unsigned long long* sumQ, double dither, uint64_t seed, uint64_t* Q) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nt; i += stride) {
        int32_t t = mesh_tris[i];
        int32_t m = obj[t];
        double n = (double)(mesh_off[m + 1] - mesh_off[m]);
        double mean = (double)sumQ[m] / n;
        double scale = dither * mean;
        uint32_t x[4];
        philox10((uint32_t)t, 0u, 0u, 1u, seed, x);
        double xi = (double)(x[0] >> 8) * (1.0 / 16777216.0);
        double d = floor(scale * xi);
        Q[i] += (uint64_t)d;
    }
}

__global__ void k_cdf_fix(const uint64_t* S, int64_t nt, const int32_t* mesh_tris, const int32_t* obj,
                          const uint32_t* mesh_off, uint64_t* cdf) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nt; i += stride) {
        int32_t m = obj[mesh_tris[i]];
        uint32_t start = mesh_off[m];
        cdf[i] = S[i] - (start > 0 ? S[start - 1] : 0ull);
    }
}

// Per canonical vertex: the distinct meshes among its incident high-curvature triangles
// (C > 0 and C >= hc_frac * max C of the mesh) each count the vertex once.
__global__ void k_hc_vertices(int64_t nv, const int32_t* canon, const uint32_t* off, const int32_t* adj,
                              const int32_t* obj, const float* C, const uint32_t* cmax_bits, float hc_frac,
                              int32_t spv, unsigned long long* ns) {
    const int lane = threadIdx.x & 31;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; v0 < nv; v0 += stride) {
        const int64_t v = v0 + lane;
        int32_t mine = -1;  // the vertex' first object; it rarely has another
        if (v < nv && canon[v] == v)
            for (uint32_t e = off[v]; e < off[v + 1]; ++e) {
                int32_t t = adj[e];
                int32_t m = obj[t];
                if (m == mine) continue;
                float thr = hc_frac * __uint_as_float(cmax_bits[m]);
                if (!(C[t] > 0.0f && C[t] >= thr)) continue;
                if (mine < 0) {
                    mine = m;
                    continue;
                }
                bool seen = false;
                for (uint32_t e2 = off[v]; e2 < e && !seen; ++e2) {
                    int32_t t2 = adj[e2];
                    if (obj[t2] != m) continue;
                    if (C[t2] > 0.0f && C[t2] >= thr) seen = true;
                }
                if (!seen) atomicAdd(&ns[m], (unsigned long long)spv);
            }
        const uint32_t same = __match_any_sync(0xffffffffu, mine);
        if (mine >= 0 && lane == __ffs(same) - 1)
            atomicAdd(&ns[mine], (unsigned long long)__popc(same) * (unsigned long long)spv);
    }
}

// (n * budget) / total without overflow (n <= total, budget < 2^63): 128-by-64 long division on 64-bit halves
__device__ __forceinline__ unsigned long long scaled_count(unsigned long long n, unsigned long long budget,
                                                           unsigned long long total) {
    const unsigned long long hi = __umul64hi(n, budget), lo = n * budget;
    unsigned long long q = 0, r = 0;
    for (int bit = 127; bit >= 0; --bit) {
        const unsigned long long b = bit >= 64 ? (hi >> (bit - 64)) & 1ull : (lo >> bit) & 1ull;
        const unsigned long long top = r >> 63;
        r = (r << 1) | b;
        if (top || r >= total) {
            r -= total;
            if (bit < 64) q |= 1ull << bit;
        }
    }
    return q;
}

// One block: empty meshes get no samples, the total is capped by the budget, offsets scanned.  Each thread takes
// the meshes tid, tid + kScThreads, ...; integer sums, so the result does not depend on the order.
constexpr int kScThreads = 1024;
__global__ void __launch_bounds__(kScThreads) k_sample_counts(int32_t n_obj, const uint32_t* mesh_off,
                                                              const uint64_t* cdf, unsigned long long* ns,
                                                              int64_t budget, int64_t* n_samples, int64_t* sample_off) {
    __shared__ unsigned long long wsum[kScThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long part = 0;
    for (int32_t m = tid; m < n_obj; m += kScThreads) {
        const uint32_t a = mesh_off[m], b = mesh_off[m + 1];
        if (b <= a || cdf[b - 1] == 0) ns[m] = 0;
        part += ns[m];
    }
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) wsum[warp] = part;
    __syncthreads();
    unsigned long long total = 0;
    for (int w = 0; w < kScThreads / 32; ++w) total += wsum[w];
    __syncthreads();  // wsum is reused by the scans below
    const bool cap = budget >= 0 && total > (unsigned long long)budget;
    int64_t carry = 0;
    for (int32_t base = 0; base < n_obj; base += kScThreads) {
        const int32_t m = base + tid;
        unsigned long long n = m < n_obj ? ns[m] : 0ull;
        if (m < n_obj && cap) n = scaled_count(n, (unsigned long long)budget, total);
        // exclusive scan over the block: within the warp, then over the warp totals
        unsigned long long x = n;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned long long before = 0, chunk = 0;
        for (int w = 0; w < kScThreads / 32; ++w) {
            if (w < warp) before += wsum[w];
            chunk += wsum[w];
        }
        if (m < n_obj) {
            n_samples[m] = (int64_t)n;
            sample_off[m] = carry + (int64_t)(before + x - n);
        }
        carry += (int64_t)chunk;
        __syncthreads();  // wsum is rewritten by the next chunk
    }
    if (tid == 0) sample_off[n_obj] = carry;
}

// ---------------------------------------------------------------- LBVH
__device__ __forceinline__ uint32_t ord(float f) {  // monotone float -> uint
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unord(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

__global__ void k_bounds(const float* V, int64_t nv, uint32_t* bnd /*[6]: lo ord, hi ord*/) {
    __shared__ uint32_t s[6];
    if (threadIdx.x < 3) s[threadIdx.x] = 0xffffffffu;
    else if (threadIdx.x < 6) s[threadIdx.x] = 0u;
    __syncthreads();
    uint32_t lo[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, hi[3] = {0, 0, 0};
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += stride)
        for (int k = 0; k < 3; ++k) {
            uint32_t o = ord(V[3 * i + k]);
            lo[k] = min(lo[k], o);
            hi[k] = max(hi[k], o);
        }
    for (int k = 0; k < 3; ++k) {
        atomicMin(&s[k], lo[k]);
        atomicMax(&s[3 + k], hi[k]);
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(&bnd[threadIdx.x], s[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&bnd[threadIdx.x], s[threadIdx.x]);
}

__device__ __forceinline__ uint64_t spread21(uint64_t x) {
    x &= 0x1fffffull;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

__global__ void k_morton(const float* V, const int32_t* T, int64_t nt, const uint32_t* bnd, uint64_t* keys,
                         uint32_t* vals) {
    float lo[3], ext[3];
    for (int k = 0; k < 3; ++k) {
        lo[k] = unord(bnd[k]);
        float hi = unord(bnd[3 + k]);
        ext[k] = hi - lo[k];
    }
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += stride) {
        uint64_t q[3];
        for (int k = 0; k < 3; ++k) {
            float c = (V[3 * (int64_t)T[3 * t] + k] + V[3 * (int64_t)T[3 * t + 1] + k]) + V[3 * (int64_t)T[3 * t + 2] + k];
            c = c * (1.0f / 3.0f);
            float u = ext[k] > 0.0f ? (c - lo[k]) / ext[k] : 0.5f;
            u = fminf(fmaxf(u, 0.0f), 1.0f);
            // 16 bits an axis: cells as fine as the boxes' padding, 1e-5 of the scene's diagonal, below which no hierarchy
            // tells triangles apart.  (21 bits took two more passes and 3 % of a build, and among 160k triangles of 2-10 cm
            // objects in scenes of 10 to 3,000 m traversal was between 0.92 and 1.05 of this.)
            uint32_t qi = (uint32_t)(u * 65535.0f);
            q[k] = qi;
        }
        keys[t] = (spread21(q[0]) << 2) | (spread21(q[1]) << 1) | spread21(q[2]);
        vals[t] = (uint32_t)t;
    }
}

// Morton keys of n points P [n][3] in the bounds bnd (the top level's instance box centres)
__global__ void k_morton_pts(const float* P, int64_t n, const uint32_t* bnd, uint64_t* keys, uint32_t* vals) {
    float lo[3], ext[3];
    for (int k = 0; k < 3; ++k) {
        lo[k] = unord(bnd[k]);
        ext[k] = unord(bnd[3 + k]) - lo[k];
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
        uint64_t q[3];
        for (int k = 0; k < 3; ++k) {
            float u = ext[k] > 0.0f ? (P[3 * t + k] - lo[k]) / ext[k] : 0.5f;
            u = fminf(fmaxf(u, 0.0f), 1.0f);
            q[k] = (uint32_t)(u * 2097151.0f);
        }
        keys[t] = (spread21(q[0]) << 2) | (spread21(q[1]) << 1) | spread21(q[2]);
        vals[t] = (uint32_t)t;
    }
}

__device__ __forceinline__ int delta(const uint64_t* k, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    uint64_t a = k[i], b = k[j];
    if (a == b) return 64 + __clz((uint32_t)(i ^ j));
    return __clzll(a ^ b);
}

// Karras (HPG 2012): internal node i covers a key range; children are leaves at the range ends.
__global__ void k_karras(const uint64_t* keys, int n, int2* child /*[n-1]: encoded (x<0 = leaf ~idx)*/,
                         int2* range, int32_t* parent_int, int32_t* parent_leaf) {
    int stride = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n - 1; i += stride) {
        int d = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
        int dmin = delta(keys, n, i, i - d);
        int lmax = 2;
        while (delta(keys, n, i, i + lmax * d) > dmin) lmax *= 2;
        int l = 0;
        for (int t = lmax / 2; t >= 1; t /= 2)
            if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
        int j = i + l * d;
        int dnode = delta(keys, n, i, j);
        int s = 0;
        int t = l;
        do {
            t = (t + 1) >> 1;
            if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
        } while (t > 1);
        int gamma = i + s * d + min(d, 0);
        int lo = min(i, j), hi = max(i, j);
        int left = (lo == gamma) ? ~gamma : gamma;
        int right = (hi == gamma + 1) ? ~(gamma + 1) : gamma + 1;
        child[i] = make_int2(left, right);
        range[i] = make_int2(lo, hi);
        if (left < 0) parent_leaf[gamma] = i; else parent_int[gamma] = i;
        if (right < 0) parent_leaf[gamma + 1] = i; else parent_int[gamma + 1] = i;
    }
}

struct Box {
    float lo[3], hi[3];
};

// leaf boxes: a triangle's vertex bounds grown by pad; an instance's world box (from its record)
struct TriLeafBox {
    const float* V;
    const int32_t* T;
    const uint32_t* sorted;
    float pad;
    __device__ __forceinline__ Box operator()(int p) const {
        const int64_t t = sorted[p];
        Box b;
        for (int k = 0; k < 3; ++k) {
            float a = V[3 * (int64_t)T[3 * t] + k], bb = V[3 * (int64_t)T[3 * t + 1] + k],
                  c = V[3 * (int64_t)T[3 * t + 2] + k];
            b.lo[k] = fminf(fminf(a, bb), c) - pad;
            b.hi[k] = fmaxf(fmaxf(a, bb), c) + pad;
        }
        return b;
    }
};
struct InstLeafBox {
    const float4* rec;
    const int32_t* sorted;
    __device__ __forceinline__ Box operator()(int p) const {
        const int64_t i = sorted[p];
        const float4 lo = rec[8 * i + 6], hi = rec[8 * i + 7];
        return Box{{lo.x, lo.y, lo.z}, {hi.x, hi.y, hi.z}};
    }
};

// ---------------------------------------------------------------- hierarchy by parallel locally-ordered clustering
// (Meister and Bittner, TVCG 2018.)  Clusters start as the triangles in Morton order; in every round each looks kPlocR
// places to either side for the neighbour whose union with it has the least surface, and clusters that choose each other
// merge.  Against the radix tree over the Morton codes (below, kept for prototypes and instances):
// closest-hit queries of a 1M-triangle clutter visit 9.4 wide nodes instead of 20.8, of a forest 29 instead
// of 57 (large triangles beside small ones spoil the radix tree's boxes), among equal leaves 58 instead of 63; the passes
// over these took 9.52 ms instead of 10.15, 2.71 instead of 3.56, 13.7 instead of 14.7.  A round is two launches; the last
// kPlocLast clusters merge in one block.  What bounds it is the chain of rounds (200k triangles: 23 of ~8 us each and one
// block's 28 in 52 us, ~0.42 ms of device time, where the radix tree with its climbs for boxes takes 0.09).
constexpr int kPlocR = 8;
constexpr int kPlocLast = 1024;       // clusters that one block merges to the end, one a thread
// Rounds can stall: of concentric shapes each prefers its smaller neighbour, and only the innermost two prefer each other.
// After a round that left more than 15 of 16 clusters (ordinary meshes: 0.73 to 0.78 of them) neighbours in order are paired
// where one lies within the other, and after another one all of them, so three rounds leave half at most.
constexpr int kPlocRounds = 320;      // of launches, and of the last block, at most: 226 of 15/16 each from 2^31 clusters
constexpr int kPlocThreads = 512;
constexpr int kPlocTile = kPlocThreads - 2 * kPlocR;  // clusters per block of a round: the others are its margins

struct PlocArgs {
    int n;                  // leaves
    int32_t* ref[2];        // clusters of even and odd rounds: leaf ~i or raw node (numbered as made)
    Box* box[2];
    int32_t* mate;          // per cluster of a round: its partner, or -1
    uint2* tiles;           // per tile of a round: clusters kept, merges
    char* scan;             // scratch of their scan
    uint32_t* count;        // [kPlocRounds + 2] clusters at the start of a round
    uint32_t* nodes;        // [kPlocRounds + 2] nodes made before it
    int2* child;            // [n - 1] raw nodes
    int32_t* size;          // [n - 1] leaves below
    int32_t* par_i;         // [n - 1], [n]
    int32_t* par_l;
    Box* box_tmp;           // [n - 1][2] the children's boxes by final node id
    uint32_t* perm_in;      // [n] the order before
    uint32_t* left;         // clusters left by the last block
};

__device__ __forceinline__ float union_area(const Box& a, const Box& b) {
    const float x = fmaxf(a.hi[0], b.hi[0]) - fminf(a.lo[0], b.lo[0]);
    const float y = fmaxf(a.hi[1], b.hi[1]) - fminf(a.lo[1], b.lo[1]);
    const float z = fmaxf(a.hi[2], b.hi[2]) - fminf(a.lo[2], b.lo[2]);
    return x * y + y * z + z * x;
}
__device__ __forceinline__ Box box_union(const Box& a, const Box& b) {
    Box u;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        u.lo[k] = fminf(a.lo[k], b.lo[k]);
        u.hi[k] = fmaxf(a.hi[k], b.hi[k]);
    }
    return u;
}
// place of the best partner of cluster i among n (box(j): its box): least area, then nearest, then the one paired with i
// by parity, so that equal clusters pair up
template <class F>
__device__ __forceinline__ int ploc_best(int i, int n, const Box& b, const F& box) {
    unsigned long long best = ~0ull;
    int at = -1;
    const int lo = max(0, i - kPlocR), hi = min(n - 1, i + kPlocR);
    for (int j = lo; j <= hi; ++j) {
        if (j == i) continue;
        const uint32_t tie = (uint32_t)(2 * abs(j - i) + (j != (i ^ 1) ? 1 : 0));
        const unsigned long long key = ((unsigned long long)__float_as_uint(union_area(b, box(j))) << 32) | tie;
        if (key < best) {
            best = key;
            at = j;
        }
    }
    return at;
}

// whether a round that found `before` clusters and left n hardly merged any
__device__ __forceinline__ bool ploc_stalled(int before, int n) { return n > before - before / 16; }
// the partner that cluster i chooses; stalls: how many of the last two rounds in a row stalled
template <class F>
__device__ __forceinline__ int ploc_choose(int i, int n, const Box& b, const F& box, int stalls) {
    const int j = i ^ 1;
    if (stalls > 0 && j < n) {
        const Box o = box(j);
        if (stalls > 1 || union_area(b, o) <= 1.125f * fmaxf(union_area(b, b), union_area(o, o))) return j;
    }
    return stalls > 1 ? -1 : ploc_best(i, n, b, box);
}

template <class LeafBox>
__global__ void k_ploc_init(const LeafBox leaf, const PlocArgs a) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
        a.ref[0][i] = ~i;
        a.box[0][i] = leaf(i);
        if (i == 0) {
            a.count[0] = (uint32_t)a.n;
            a.nodes[0] = 0u;
            a.par_i[a.n - 2] = -1;  // the last node made is the root
        }
    }
}

// raw node id of clusters l and r: their boxes bl and br, together so many leaves
__device__ __forceinline__ void ploc_node(const PlocArgs& a, int id, int32_t l, int32_t r, const Box& bl, const Box& br,
                                          int32_t size) {
    a.child[id] = make_int2(l, r);
    a.size[id] = size;
    if (l < 0) a.par_l[~l] = id; else a.par_i[l] = id;
    if (r < 0) a.par_l[~r] = id; else a.par_i[r] = id;
    const int fin = a.n - 2 - id;
    a.box_tmp[2 * fin] = bl;
    a.box_tmp[2 * fin + 1] = br;
}

// A block looks up the neighbours chosen by its tile's clusters and by kPlocR to either side, so that it knows who of the
// tile was chosen back: partners and the tile's counts in one launch.
__global__ void __launch_bounds__(kPlocThreads) k_ploc_mate(const PlocArgs a, int it) {
    __shared__ Box t[kPlocThreads + 2 * kPlocR];
    __shared__ int32_t nn[kPlocThreads];
    const int n = (int)a.count[it], base = (int)blockIdx.x * kPlocTile;
    if (base >= n) return;
    const bool stalled = it > 0 && ploc_stalled((int)a.count[it - 1], n);
    const int stalls = !stalled ? 0 : it > 1 && ploc_stalled((int)a.count[it - 2], (int)a.count[it - 1]) ? 2 : 1;
    const Box* box = it & 1 ? a.box[1] : a.box[0];
    for (int e = threadIdx.x; e < kPlocThreads + 2 * kPlocR; e += kPlocThreads) {
        const int i = base - 2 * kPlocR + e;
        if (i >= 0 && i < n) t[e] = box[i];
    }
    __syncthreads();
    const int at = base - kPlocR, i = at + (int)threadIdx.x;  // nn[e]: chosen by cluster at + e
    auto boxes = [&](int j) { return t[j - at + kPlocR]; };
    nn[threadIdx.x] = i >= 0 && i < n ? ploc_choose(i, n, t[threadIdx.x + kPlocR], boxes, stalls) : -1;
    __syncthreads();
    uint32_t kept = 0, merged = 0;
    if (i >= base && i < base + kPlocTile && i < n) {
        const int j = nn[threadIdx.x];  // within kPlocR of i, so nn[j - at] is there
        const bool both = j >= 0 && nn[j - at] == i;
        a.mate[i] = both ? j : -1;
        kept = !both || i < j;
        merged = both && i < j;
    }
    const int kept_all = __syncthreads_count(kept), merged_all = __syncthreads_count(merged);
    if (threadIdx.x == 0) a.tiles[blockIdx.x] = make_uint2((uint32_t)kept_all, (uint32_t)merged_all);
}

// exclusive scan over the block of a pair of counts (s: one pair per warp); *total: the block's sums
__device__ __forceinline__ uint2 block_excl2(uint2 v, uint2* s, int warps, uint2* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint2 x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t p = __shfl_up_sync(0xffffffffu, x.x, o), q = __shfl_up_sync(0xffffffffu, x.y, o);
        if (lane >= o) {
            x.x += p;
            x.y += q;
        }
    }
    if (lane == 31) s[warp] = x;
    __syncthreads();
    uint2 before = make_uint2(0u, 0u), all = make_uint2(0u, 0u);
    for (int w = 0; w < warps; ++w) {
        const uint2 c = s[w];
        if (w < warp) {
            before.x += c.x;
            before.y += c.y;
        }
        all.x += c.x;
        all.y += c.y;
    }
    __syncthreads();
    *total = all;
    return make_uint2(before.x + x.x - v.x, before.y + x.y - v.y);
}

// SCANNED: a.tiles hold the sums up to and with each tile, else a block adds up the tiles before it itself, which grows with
// the square of the clusters (kPlocSelf tiles, 4M clusters: 0.3 GB of reads from L2)
constexpr int kPlocSelf = 8192;
template <bool SCANNED>
__global__ void __launch_bounds__(kPlocThreads) k_ploc_merge(const PlocArgs a, int it) {
    constexpr int kWarps = kPlocThreads / 32;
    __shared__ uint2 s[kWarps];
    const int n = (int)a.count[it], base = (int)blockIdx.x * kPlocTile;
    if (base >= n) return;
    uint2 pre = make_uint2(0u, 0u), own = make_uint2(0u, 0u), before, total;
    if (SCANNED) {
        if (threadIdx.x == 0 && blockIdx.x > 0) pre = a.tiles[blockIdx.x - 1];
    } else {
        for (int b = threadIdx.x; b < (int)blockIdx.x; b += kPlocThreads) {
            const uint2 t = a.tiles[b];
            pre.x += t.x;
            pre.y += t.y;
        }
    }
    const int i = base + (int)threadIdx.x;
    const bool live = (int)threadIdx.x < kPlocTile && i < n;
    const int j = live ? a.mate[i] : -1;
    own.x = live && (j < 0 || i < j);
    own.y = live && j >= 0 && i < j;
    block_excl2(pre, s, kWarps, &before);  // sums of the tiles before this one
    const uint2 at = block_excl2(own, s, kWarps, &total);
    const uint32_t first = a.nodes[it];
    if (threadIdx.x == 0 && base + kPlocTile >= n) {
        a.count[it + 1] = before.x + total.x;
        a.nodes[it + 1] = first + before.y + total.y;
    }
    if (!own.x) return;
    const int32_t* ref = it & 1 ? a.ref[1] : a.ref[0];
    const Box* box = it & 1 ? a.box[1] : a.box[0];
    const uint32_t pos = before.x + at.x;
    int32_t r = ref[i];
    Box b = box[i];
    if (own.y) {
        const int id = (int)(first + before.y + at.y);
        const int32_t r2 = ref[j];
        const Box b2 = box[j];
        ploc_node(a, id, r, r2, b, b2, (r < 0 ? 1 : a.size[r]) + (r2 < 0 ? 1 : a.size[r2]));
        r = id;
        b = box_union(b, b2);
    }
    (it & 1 ? a.ref[0] : a.ref[1])[pos] = r;
    (it & 1 ? a.box[0] : a.box[1])[pos] = b;
}

// The last clusters (at most kPlocLast), a thread each, rounds in one block; *a.left: clusters left (1, or all of them if
// they are more).  About 28 dependent rounds: boxes, ids and sizes stay in shared memory, and one packed scan places
// both the clusters kept (low half) and the nodes made.
__global__ void __launch_bounds__(kPlocLast) k_ploc_last(const PlocArgs a, int it) {
    __shared__ Box box[kPlocLast];
    __shared__ int32_t ref[kPlocLast], sizes[kPlocLast], nn[kPlocLast];
    __shared__ uint32_t sums[kPlocLast / 32];
    int n = (int)a.count[it];
    int base = (int)a.nodes[it];
    if (n > kPlocLast) {
        if (threadIdx.x == 0) *a.left = (uint32_t)n;
        return;
    }
    const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
    int32_t r = 0, size = 0;
    Box b{};
    if (i < n) {
        box[i] = b = (it & 1 ? a.box[1] : a.box[0])[i];
        ref[i] = r = (it & 1 ? a.ref[1] : a.ref[0])[i];
        sizes[i] = size = r < 0 ? 1 : a.size[r];
    }
    __syncthreads();
    int stalls = 0;
    for (int round = 0; n > 1 && round < kPlocRounds; ++round) {
        if (i < n) nn[i] = ploc_choose(i, n, b, [&](int j) { return box[j]; }, stalls);
        __syncthreads();
        const int j = i < n ? nn[i] : -1;
        const bool both = j >= 0 && nn[j] == i, join = both && i < j, keep = i < n && (!both || join);
        Box b2{};
        int32_t r2 = 0, size2 = 0;
        if (join) {
            b2 = box[j];
            r2 = ref[j];
            size2 = sizes[j];
        }
        const uint32_t km = __ballot_sync(0xffffffffu, keep), jm = __ballot_sync(0xffffffffu, join);
        if (lane == 0) sums[warp] = (uint32_t)__popc(km) | ((uint32_t)__popc(jm) << 16);
        __syncthreads();  // (also between the reads above and the writes below)
        const uint32_t w = sums[lane], all = __reduce_add_sync(0xffffffffu, w),
                       before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
        const uint32_t below = (1u << lane) - 1u;
        const int pos = (int)(before & 0xffffu) + __popc(km & below);
        if (join) {
            const int id = base + (int)(before >> 16) + __popc(jm & below);
            size += size2;
            ploc_node(a, id, r, r2, b, b2, size);
            r = id;
            b = box_union(b, b2);
        }
        if (keep) {
            box[pos] = b;
            ref[pos] = r;
            sizes[pos] = size;
        }
        stalls = ploc_stalled(n, (int)(all & 0xffffu)) ? min(stalls + 1, 2) : 0;
        n = (int)(all & 0xffffu);
        base += (int)(all >> 16);
        __syncthreads();
        if (i < n) {
            b = box[i];
            r = ref[i];
            size = sizes[i];
        }
    }
    if (threadIdx.x == 0) *a.left = (uint32_t)n;
}

// the hierarchy in the radix tree's form: node ids from the root (0), leaves in depth-first order (a node's leaves are
// a range), which permutes the triangles
__global__ void k_ploc_layout(const PlocArgs a, uint32_t* perm, int32_t* pos_of) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < a.n; p += gridDim.x * blockDim.x) {
        int pos = 0, self = ~p;
        int node = a.par_l[p];
        for (int climb = 0; node >= 0 && climb < a.n; ++climb) {
            const int2 c = a.child[node];
            if (c.y == self) pos += c.x < 0 ? 1 : a.size[c.x];
            self = node;
            node = a.par_i[node];
        }
        pos_of[p] = pos;
        perm[pos] = a.perm_in[p];
    }
}

__global__ void k_ploc_emit(const PlocArgs a, const int32_t* pos_of, int2* child, int2* range, int32_t* out_par_i,
                            int32_t* out_par_l) {
    const int root = a.n - 2;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n - 1; i += gridDim.x * blockDim.x) {
        const int id = root - i;
        const int2 c = a.child[i];
        int first = i;  // the node's first leaf, down its left side
        for (int down = 0; first >= 0 && down < a.n; ++down) first = a.child[first].x;
        const int lo = pos_of[~first];
        range[id] = make_int2(lo, lo + a.size[i] - 1);
        const int l = c.x < 0 ? ~pos_of[~c.x] : root - c.x, r = c.y < 0 ? ~pos_of[~c.y] : root - c.y;
        child[id] = make_int2(l, r);
        if (l < 0) out_par_l[~l] = id; else out_par_i[l] = id;
        if (r < 0) out_par_l[~r] = id; else out_par_i[r] = id;
    }
}

// Bottom-up boxes: each leaf writes its box into its parent's slot; the second child to arrive at
// a node unites both slots and climbs.  box_tmp: [n-1][2] boxes.
template <class LeafBox>
__global__ void k_boxes(const LeafBox leaf, int n, const int2* child, const int32_t* parent_int,
                        const int32_t* parent_leaf, Box* box_tmp, uint32_t* visits, uint32_t* err) {
    int stride = gridDim.x * blockDim.x;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
        const Box b = leaf(p);
        int node = parent_leaf[p];
        int slot = (child[node].x == ~p) ? 0 : 1;
        box_tmp[2 * node + slot] = b;
        for (int climb = 0;; ++climb) {
            if (climb > n) {  // deeper than the node count: not a tree
                atomicOr(err, kFlagBadTree);
                break;
            }
            __threadfence();
            uint32_t old = atomicAdd(&visits[node], 1u);
            if (old == 0) break;
            if (old > 1) {  // a node has two children: a third arrival means a malformed hierarchy
                atomicOr(err, kFlagBadTree);
                break;
            }
            __threadfence();
            const volatile float* b0 = reinterpret_cast<const volatile float*>(&box_tmp[2 * node]);
            const volatile float* b1 = reinterpret_cast<const volatile float*>(&box_tmp[2 * node + 1]);
            Box u;
            for (int k = 0; k < 3; ++k) {
                u.lo[k] = fminf(b0[k], b1[k]);
                u.hi[k] = fmaxf(b0[3 + k], b1[3 + k]);
            }
            if (node == 0) break;
            int par = parent_int[node];
            int s2 = (child[par].x == node) ? 0 : 1;
            volatile float* dst = reinterpret_cast<volatile float*>(&box_tmp[2 * par + s2]);
            for (int k = 0; k < 3; ++k) {
                dst[k] = u.lo[k];
                dst[3 + k] = u.hi[k];
            }
            node = par;
        }
    }
}

__host__ __device__ __forceinline__ int32_t leaf_ref(int first, int count) { return ~((first << 3) | (count - 1)); }

// child reference of binary node i's side c: a leaf code for single triangles and for subtrees of at
// most kLeafMax triangles (a contiguous range of the leaf order), else the internal node index
__device__ __forceinline__ int32_t child_ref(int32_t cc, const int2* range, int32_t leaf_off) {
    if (cc < 0) return leaf_ref(~cc + leaf_off, 1);
    const int2 r = range[cc];
    const int cnt = r.y - r.x + 1;
    return cnt <= kLeafMax ? leaf_ref(r.x + leaf_off, cnt) : cc;
}

// Binary internal nodes that stay internal (range above kLeafMax, or the root) at even depth become
// the nodes of the 4-wide BVH: each takes its children, with internal children replaced by theirs.
__global__ void k_wide_flags(int n, const int2* range, const int32_t* parent_int, uint32_t* flag, uint32_t* err) {
    int stride = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n - 1; i += stride) {
        const int2 r = range[i];
        const bool internal = i == 0 || r.y - r.x + 1 > kLeafMax;
        uint32_t f = 0;
        if (internal) {
            int d = 0, x = i;
            while (x != 0) {
                x = parent_int[x];
                if (++d > n) {  // deeper than the node count: not a tree
                    atomicOr(err, kFlagBadTree);
                    break;
                }
            }
            f = (d & 1) == 0 ? 1u : 0u;
        }
        flag[i] = f;
    }
}

// nodes: the first node of this hierarchy; stored node references are offset by node_off and leaf codes'
// first triangles by leaf_off (several hierarchies in one array)
__global__ void k_pack_wide(int n, const int2* child, const int2* range, const Box* box_tmp, const uint32_t* flag,
                            const uint32_t* idx, float4* nodes, int32_t node_off, int32_t leaf_off) {
    int stride = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n - 1; i += stride) {
        if (!flag[i]) continue;
        float lo[3][4], hi[3][4];
        int32_t ref[4];
        int cnt = 0;
        auto add = [&](const Box& b, int32_t r) {
            for (int k = 0; k < 3; ++k) {
                lo[k][cnt] = b.lo[k];
                hi[k][cnt] = b.hi[k];
            }
            ref[cnt++] = r;
        };
        const int2 c = child[i];
        const int32_t cs[2] = {c.x, c.y};
        const int32_t self = (int32_t)idx[i] + node_off;
        for (int sd = 0; sd < 2; ++sd) {
            const int32_t r = child_ref(cs[sd], range, leaf_off);
            if (r < 0) {
                add(box_tmp[2 * i + sd], r);
            } else {
                const int2 g = child[r];
                const int32_t gs[2] = {g.x, g.y};
                for (int t = 0; t < 2; ++t) {
                    const int32_t rg = child_ref(gs[t], range, leaf_off);
                    if (rg >= 0)  // row 7 of a child node: its parent and its slot here (the stackless walk)
                        nodes[8 * (size_t)idx[rg] + 7] = make_float4(__int_as_float(self), __int_as_float(cnt), 0.0f,
                                                                     0.0f);
                    add(box_tmp[2 * r + t], rg < 0 ? rg : (int32_t)idx[rg] + node_off);
                }
            }
        }
        for (; cnt < 4; ++cnt) {
            for (int k = 0; k < 3; ++k) {
                lo[k][cnt] = 0.0f;
                hi[k][cnt] = 0.0f;
            }
            ref[cnt] = kEmptyRef;
        }
        float4* o = nodes + 8 * (size_t)idx[i];
        for (int k = 0; k < 3; ++k) {
            o[2 * k] = make_float4(lo[k][0], lo[k][1], lo[k][2], lo[k][3]);
            o[2 * k + 1] = make_float4(hi[k][0], hi[k][1], hi[k][2], hi[k][3]);
        }
        o[6] = make_float4(__int_as_float(ref[0]), __int_as_float(ref[1]), __int_as_float(ref[2]),
                           __int_as_float(ref[3]));
        if (i == 0) o[7] = make_float4(__int_as_float(-1), 0.0f, 0.0f, 0.0f);  // the root has no parent
    }
}

__global__ void k_reorder(const float* V, const int32_t* T, int64_t nt, const uint32_t* sorted_tri, float4* tri_v) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nt; p += stride) {
        int64_t t = sorted_tri[p];
        const float* a = V + 3 * (int64_t)T[3 * t];
        const float* b = V + 3 * (int64_t)T[3 * t + 1];
        const float* c = V + 3 * (int64_t)T[3 * t + 2];
        tri_v[3 * p + 0] = make_float4(a[0], a[1], a[2], __int_as_float((int32_t)t));
        tri_v[3 * p + 1] = make_float4(b[0], b[1], b[2], 0.0f);
        tri_v[3 * p + 2] = make_float4(c[0], c[1], c[2], 0.0f);
    }
}

}  // namespace

// One allocation cut into pieces.  A build needs some 30 arrays of scratch; allocating and freeing each took about 35 us,
// which was as long as the build's kernels.
struct Pieces {
    size_t bytes = 0;
    char* base = nullptr;  // null: only adds up
    template <class T>
    T* take(size_t count) {
        const size_t at = bytes;
        bytes += (count * sizeof(T) + 255) & ~size_t(255);
        return base ? reinterpret_cast<T*>(base + at) : nullptr;
    }
};

static PlocArgs ploc_pieces(Pieces& m, int n, Box* box_tmp) {
    PlocArgs a{};
    a.n = n;
    for (int k = 0; k < 2; ++k) {
        a.ref[k] = m.take<int32_t>(n);
        a.box[k] = m.take<Box>(n);
    }
    a.mate = m.take<int32_t>(n);
    a.tiles = m.take<uint2>((n + kPlocTile - 1) / kPlocTile);
    a.scan = m.take<char>(scan_scratch_bytes((n + kPlocTile - 1) / kPlocTile));
    a.count = m.take<uint32_t>(kPlocRounds + 2);
    a.nodes = m.take<uint32_t>(kPlocRounds + 2);
    a.left = m.take<uint32_t>(1);
    a.child = m.take<int2>(n);
    a.size = m.take<int32_t>(n);
    a.par_i = m.take<int32_t>(n);
    a.par_l = m.take<int32_t>(n);
    a.perm_in = m.take<uint32_t>(n);
    a.box_tmp = box_tmp;
    return a;
}

// Clustered hierarchy over n leaves in the order perm (permuted to the new leaf order): children, ranges and parents in the
// radix tree's form, and the boxes.
template <class LeafBox>
static cudaError_t ploc_build(const LeafBox& leaf, const PlocArgs& a, uint32_t* perm, int2* child, int2* range,
                              int32_t* par_i, int32_t* par_l, cudaStream_t s) {
    const int n = a.n, tiles = (n + kPlocTile - 1) / kPlocTile;
    note_launch();
    k_ploc_init<<<grid_for(n, kB), kB, 0, s>>>(leaf, a);
    CK(cudaGetLastError());
    // a round leaves 0.73 to 0.78 of the clusters: rounds for 0.79, then the count is read, and more follow if need be
    int it = 0;
    uint32_t h_left = (uint32_t)n;
    for (;;) {
        int more = 0;
        for (double c = h_left; c > kPlocLast && it + more < kPlocRounds; c *= 0.79) ++more;
        double left = h_left;
        for (int r = 0; r < more; ++r, ++it, left *= 0.79) {
            note_launch();
            k_ploc_mate<<<(unsigned)tiles, kPlocThreads, 0, s>>>(a, it);
            CK(cudaGetLastError());
            // (both counts of a tile as one 64-bit word: the sums of either stay below 2^32)
            const bool scanned = left > (double)kPlocSelf * kPlocTile;
            if (scanned) {
                uint64_t* t64 = reinterpret_cast<uint64_t*>(a.tiles);
                CK(inclusive_scan_u64(t64, t64, tiles, a.scan, s));
            }
            note_launch();
            if (scanned) k_ploc_merge<true><<<(unsigned)tiles, kPlocThreads, 0, s>>>(a, it);
            else k_ploc_merge<false><<<(unsigned)tiles, kPlocThreads, 0, s>>>(a, it);
            CK(cudaGetLastError());
        }
        note_launch();
        k_ploc_last<<<1, kPlocLast, 0, s>>>(a, it);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(&h_left, a.left, 4, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        if (h_left <= (uint32_t)kPlocLast || it >= kPlocRounds) break;
    }
    if (h_left != 1) return cudaErrorUnknown;  // (not reached: the bounds above)
    CK(cudaMemcpyAsync(a.perm_in, perm, (size_t)n * 4, cudaMemcpyDeviceToDevice, s));
    note_launch();
    k_ploc_layout<<<grid_for(n, kB), kB, 0, s>>>(a, perm, a.mate);
    CK(cudaGetLastError());
    note_launch();
    k_ploc_emit<<<grid_for(n, kB), kB, 0, s>>>(a, a.mate, child, range, par_i, par_l);
    return cudaGetLastError();
}

static cudaError_t build_two_level(SceneDev& S, float pad_world, uint32_t* flags, cudaStream_t s);

cudaError_t scene_build(SceneDev& S, const CurvParamsDev& cp, cudaStream_t s, bool* mesh_error, std::string* msg,
                        bool refit, bool keep_curvature, DevBuf* kept) {
    *mesh_error = false;
    refit = refit && (S.two_level ? S.tl_ready : S.bvh_ready);
    keep_curvature = keep_curvature && refit;
    const int64_t nv = S.n_verts, nt = S.n_tris;
    const float* V = ptr<float>(S.verts);
    const int32_t* T = ptr<int32_t>(S.tris);
    const int32_t* obj = ptr<int32_t>(S.tri_obj);
    // A refit that keeps the curvature is a handful of launches, so its scratch (52 bytes a triangle) stays with the caller:
    // whether an allocation found room in the driver's pages or mapped new ones made it 150 or 310 us at 8,000 triangles.
    DevBuf flags, own;
    DevBuf& scratch = keep_curvature && kept ? *kept : own;
    struct Guard {
        DevBuf &a, &b;
        ~Guard() {
            release(a);
            release(b);
        }
    } guard{flags, own};
    CK(grow(flags, 16));
    CK(cudaMemsetAsync(flags.p, 0, 16, s));
    note_launch();
    k_validate<<<grid_for(nv + nt, kB), kB, 0, s>>>(V, nv, T, nt, ptr<int32_t>(S.tri_mat), S.n_mat, obj,
                                                    ptr<uint32_t>(flags));
    CK(cudaGetLastError());
    uint32_t hflags = 0;
    CK(cudaMemcpyAsync(&hflags, flags.p, 4, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hflags) {
        *mesh_error = true;
        *msg = (hflags & kFlagBadVertex) ? "non-finite vertex coordinate" : "triangle index, material or object out of range";
        return cudaSuccess;
    }
    // ---- scratch: one allocation (its sizes are known once the mesh is found valid), freed at the end of the build
    const int32_t n_obj = S.n_obj;  // known from the host copy
    const int64_t nmax = std::max<int64_t>(std::max<int64_t>(nv, nt), 1);
    const bool curv = !keep_curvature, flat = !S.two_level && nt > kLeafMax;
    const bool sorts = curv || (!refit && !S.two_level);
    struct Scratch {
        uint32_t *bnd, *vals, *cnt, *off, *cursor, *cmax, *moff, *visits, *wtotal;
        uint64_t *keys, *Q, *S64;
        unsigned long long *sumQ, *nsu;
        int32_t *canon, *adj;
        float* Gc;
        char *sort_scr, *wscan_scr;
        Box* boxes;
        PlocArgs ploc;
    } w{};
    auto lay = [&](Pieces m) {
        w.bnd = m.take<uint32_t>(16);
        if (sorts) {
            w.keys = m.take<uint64_t>(nmax);
            w.vals = m.take<uint32_t>(nmax);
            w.sort_scr = m.take<char>(sort_scratch_bytes(nmax) + scan_scratch_bytes(nmax + n_obj + 1));
        }
        if (curv) {
            w.canon = m.take<int32_t>(nv);
            w.cnt = m.take<uint32_t>(std::max<int64_t>(nv, n_obj) + 1);
            w.off = m.take<uint32_t>(nv + 1);
            w.cursor = m.take<uint32_t>(nv + 1);
            w.adj = m.take<int32_t>(std::max<int64_t>(3 * nt, 1));
            w.Gc = m.take<float>(nv);
            w.cmax = m.take<uint32_t>(n_obj + 1);
            w.moff = m.take<uint32_t>(n_obj + 2);
            w.sumQ = m.take<unsigned long long>(n_obj + 1);
            w.Q = m.take<uint64_t>(nmax);
            w.S64 = m.take<uint64_t>(nmax);
            w.nsu = m.take<unsigned long long>(n_obj + 1);
        }
        if (flat) {
            w.boxes = m.take<Box>(2 * (nt - 1));
            w.visits = m.take<uint32_t>(nt - 1);
            if (!refit) {
                w.wscan_scr = m.take<char>(scan_scratch_bytes(nt - 1));
                w.wtotal = m.take<uint32_t>(1);
                w.ploc = ploc_pieces(m, (int)nt, w.boxes);
            }
        }
        return m.bytes;
    };
    CK(grow(scratch, lay(Pieces{})));
    lay(Pieces{0, ptr<char>(scratch)});
    uint32_t* keys32 = reinterpret_cast<uint32_t*>(w.keys);  // (the 32-bit sorts' keys)

    CK(grow(S.nrm, (size_t)nt * 3 * sizeof(float)));
    note_launch();
    k_normals<<<grid_for(nt, kB), kB, 0, s>>>(V, T, nt, ptr<float>(S.nrm));
    CK(cudaGetLastError());

    if (!keep_curvature) {
        // ---- weld
        note_launch();
        k_pos_keys<<<grid_for(nv, kB), kB, 0, s>>>(V, nv, keys32, w.vals);
        CK(cudaGetLastError());
        CK(radix_sort_u32(keys32, w.vals, nv, 0, 32, w.sort_scr, s));
        note_launch();
        k_weld_runs<<<grid_for(nv, kB), kB, 0, s>>>(V, nv, keys32, w.vals, w.canon);
        CK(cudaGetLastError());

        // ---- adjacency CSR over canonical vertices
        CK(cudaMemsetAsync(w.cnt, 0, (size_t)(nv + 1) * 4, s));
        CK(cudaMemsetAsync(w.cursor, 0, (size_t)(nv + 1) * 4, s));
        note_launch();
        k_adj_count<<<grid_for(nt, kB), kB, 0, s>>>(w.canon, T, nt, w.cnt);
        CK(cudaGetLastError());
        CK(exclusive_scan_u32(w.cnt, w.off, nv + 1, nullptr, w.sort_scr, s));
        note_launch();
        k_adj_fill<<<grid_for(nt, kB), kB, 0, s>>>(w.canon, T, nt, w.off, w.cursor,
                                                  w.adj);
        CK(cudaGetLastError());
        note_launch();
        k_adj_sort<<<grid_for(nv, kB), kB, 0, s>>>(nv, w.off, w.adj);
        CK(cudaGetLastError());

        // ---- curvature and metric
        CK(grow(S.G, (size_t)nv * 4));
        CK(grow(S.C, (size_t)nt * 4));
        note_launch();
        k_curvature<<<grid_for(nv, kB), kB, 0, s>>>(V, nv, T, w.canon, w.off, w.adj,
                                                   w.Gc);
        CK(cudaGetLastError());
        note_launch();
        k_expand_G<<<grid_for(nv, kB), kB, 0, s>>>(w.canon, nv, w.Gc, ptr<float>(S.G));
        CK(cudaGetLastError());
        CK(cudaMemsetAsync(w.cmax, 0, (size_t)(n_obj + 1) * 4, s));
        note_launch();
        k_metric<<<grid_for(nt, kB), kB, 0, s>>>(V, T, nt, w.canon, ptr<float>(S.G), cp.eta, cp.area_ref,
                                                ptr<float>(S.C), w.cmax, obj);
        CK(cudaGetLastError());

        // ---- per-mesh triangle lists (ascending), integer weights, CDFs
        CK(cudaMemsetAsync(w.cnt, 0, (size_t)(n_obj + 1) * 4, s));
        note_launch();
        k_mesh_count<<<grid_for(nt, kB), kB, 0, s>>>(obj, nt, w.cnt);
        CK(cudaGetLastError());
        CK(exclusive_scan_u32(w.cnt, w.moff, n_obj + 1, nullptr, w.sort_scr, s));
        CK(grow(S.mesh_tris, (size_t)nt * 4));
        {
            // triangles grouped by mesh, ascending inside a mesh (the sort is stable)
            int mesh_bits = 1;
            while ((1ll << mesh_bits) <= (int64_t)n_obj) ++mesh_bits;
            note_launch();
            k_mesh_keys<<<grid_for(nt, kB), kB, 0, s>>>(obj, nt, keys32, w.vals);
            CK(cudaGetLastError());
            CK(radix_sort_u32(keys32, w.vals, nt, 0, mesh_bits, w.sort_scr, s));
            CK(cudaMemcpyAsync(S.mesh_tris.p, w.vals, (size_t)nt * 4, cudaMemcpyDeviceToDevice, s));
        }
        CK(cudaMemsetAsync(w.sumQ, 0, (size_t)(n_obj + 1) * 8, s));
        note_launch();
        k_quantize<<<grid_for(nt, kB), kB, 0, s>>>(ptr<int32_t>(S.mesh_tris), nt, obj, ptr<float>(S.C), w.cmax,
                                                  w.Q, w.sumQ);
        CK(cudaGetLastError());
        note_launch();
        k_dither<<<grid_for(nt, kB), kB, 0, s>>>(ptr<int32_t>(S.mesh_tris), nt, obj, w.moff,
                                                w.sumQ, cp.dither, cp.seed, w.Q);
        CK(cudaGetLastError());
        CK(inclusive_scan_u64(w.Q, w.S64, nt, w.sort_scr, s));
        CK(grow(S.cdf, (size_t)nt * 8));
        note_launch();
        k_cdf_fix<<<grid_for(nt, kB), kB, 0, s>>>(w.S64, nt, ptr<int32_t>(S.mesh_tris), obj,
                                                 w.moff, ptr<uint64_t>(S.cdf));
        CK(cudaGetLastError());
        // mesh offsets as int64 for the sampling kernels
        CK(grow(S.mesh_off, (size_t)(n_obj + 1) * 8));
        note_launch();
        k_widen<<<grid_for(n_obj + 1, kB), kB, 0, s>>>(w.moff, n_obj + 1, ptr<int64_t>(S.mesh_off));
        CK(cudaGetLastError());
        // sample counts
        CK(cudaMemsetAsync(w.nsu, 0, (size_t)(n_obj + 1) * 8, s));
        note_launch();
        k_hc_vertices<<<grid_for(nv, kB), kB, 0, s>>>(nv, w.canon, w.off, w.adj, obj,
                                                     ptr<float>(S.C), w.cmax, cp.hc_frac,
                                                     cp.samples_per_vertex, w.nsu);
        CK(cudaGetLastError());
        CK(grow(S.n_samples, (size_t)(n_obj + 1) * 8));
        CK(grow(S.sample_off, (size_t)(n_obj + 1) * 8));
        note_launch();
        k_sample_counts<<<1, kScThreads, 0, s>>>(n_obj, w.moff, ptr<uint64_t>(S.cdf), w.nsu,
                                        cp.budget, ptr<int64_t>(S.n_samples), ptr<int64_t>(S.sample_off));
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(&S.total_samples, ptr<int64_t>(S.sample_off) + n_obj, 8, cudaMemcpyDeviceToHost, s));

    }  // !keep_curvature

    // ---- hierarchy
    {
        uint32_t init[6] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u};
        CK(cudaMemcpyAsync(w.bnd, init, sizeof(init), cudaMemcpyHostToDevice, s));
    }
    note_launch();
    k_bounds<<<grid_for(nv, kB, 152 * 4), kB, 0, s>>>(V, nv, w.bnd);
    CK(cudaGetLastError());
    if (!refit && !S.two_level) {
        note_launch();
        k_morton<<<grid_for(nt, kB), kB, 0, s>>>(V, T, nt, w.bnd, w.keys, w.vals);
        CK(cudaGetLastError());
        CK(radix_sort_u64(w.keys, w.vals, nt, 48, w.sort_scr, s));
        CK(grow(S.bvh_perm, (size_t)nt * 4));
        CK(cudaMemcpyAsync(S.bvh_perm.p, w.vals, (size_t)nt * 4, cudaMemcpyDeviceToDevice, s));
    }
    uint32_t hb[6];
    CK(cudaMemcpyAsync(hb, w.bnd, sizeof(hb), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    {
        double diag2 = 0;
        for (int k = 0; k < 3; ++k) {
            auto un = [](uint32_t u) {
                uint32_t b = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
                float f;
                memcpy(&f, &b, 4);
                return f;
            };
            S.bounds_lo[k] = un(hb[k]);
            S.bounds_hi[k] = un(hb[3 + k]);
            double e = (double)S.bounds_hi[k] - S.bounds_lo[k];
            diag2 += e * e;
        }
        const float pad = (float)(1e-5 * sqrt(diag2) + 1e-7);
        const int n = (int)nt;
        if (S.two_level) {
            // no hierarchy over the world triangles: the prototypes' BVHs and one over the instances
            for (DevBuf* b : {&S.tri_v, &S.bvh_child, &S.bvh_range, &S.bvh_par_i, &S.bvh_par_l, &S.bvh_perm,
                              &S.bvh_wflag, &S.bvh_widx})
                release(*b);
            S.bvh_ready = false;
            CK(build_two_level(S, pad, ptr<uint32_t>(flags), s));
        } else {
            S.tl_ready = false;
            CK(grow(S.tri_v, (size_t)nt * 3 * sizeof(float4)));
            if (n == 1 || n <= kLeafMax) {
                CK(grow(S.nodes, 8 * sizeof(float4)));
                S.root = leaf_ref(0, n);
            } else {
                S.root = 0;
                int2* child_p = ptr<int2>(S.bvh_child);
                int2* range_p = ptr<int2>(S.bvh_range);
                if (!refit) {
                    CK(grow(S.bvh_child, (size_t)(n - 1) * sizeof(int2)));
                    CK(grow(S.bvh_range, (size_t)(n - 1) * sizeof(int2)));
                    CK(grow(S.bvh_par_i, (size_t)n * 4));
                    CK(grow(S.bvh_par_l, (size_t)n * 4));
                    child_p = ptr<int2>(S.bvh_child);
                    range_p = ptr<int2>(S.bvh_range);
                    CK(ploc_build(TriLeafBox{V, T, ptr<uint32_t>(S.bvh_perm), pad}, w.ploc, ptr<uint32_t>(S.bvh_perm),
                                  child_p, range_p, ptr<int32_t>(S.bvh_par_i), ptr<int32_t>(S.bvh_par_l), s));
                } else {
                    CK(cudaMemsetAsync(w.visits, 0, (size_t)(n - 1) * 4, s));
                    note_launch();
                    k_boxes<<<grid_for(n, kB), kB, 0, s>>>(TriLeafBox{V, T, ptr<uint32_t>(S.bvh_perm), pad}, n, child_p,
                                                           ptr<int32_t>(S.bvh_par_i), ptr<int32_t>(S.bvh_par_l),
                                                           w.boxes, w.visits, ptr<uint32_t>(flags));
                    CK(cudaGetLastError());
                }
                if (!refit) {
                    // 4-wide BVH: flag the binary nodes that become wide nodes, number them
                    CK(grow(S.bvh_wflag, (size_t)(n - 1) * 4));
                    CK(grow(S.bvh_widx, (size_t)(n - 1) * 4));
                    note_launch();
                    k_wide_flags<<<grid_for(n - 1, kB), kB, 0, s>>>(n, range_p, ptr<int32_t>(S.bvh_par_i),
                                                                    ptr<uint32_t>(S.bvh_wflag), ptr<uint32_t>(flags));
                    CK(cudaGetLastError());
                    CK(exclusive_scan_u32(ptr<uint32_t>(S.bvh_wflag), ptr<uint32_t>(S.bvh_widx), n - 1,
                                          w.wtotal, w.wscan_scr, s));
                    uint32_t n4 = 0;
                    CK(cudaMemcpyAsync(&n4, w.wtotal, 4, cudaMemcpyDeviceToHost, s));
                    CK(cudaStreamSynchronize(s));
                    CK(grow(S.nodes, (size_t)std::max<uint32_t>(n4, 1) * 8 * sizeof(float4)));
                    S.n_nodes = n4;
                }
                note_launch();
                k_pack_wide<<<grid_for(n - 1, kB), kB, 0, s>>>(n, child_p, range_p, w.boxes,
                                                               ptr<uint32_t>(S.bvh_wflag), ptr<uint32_t>(S.bvh_widx),
                                                               ptr<float4>(S.nodes), 0, 0);
                CK(cudaGetLastError());
            }
            note_launch();
            k_reorder<<<grid_for(nt, kB), kB, 0, s>>>(V, T, nt, ptr<uint32_t>(S.bvh_perm), ptr<float4>(S.tri_v));
            CK(cudaGetLastError());
        }
    }
    CK(cudaMemcpyAsync(&hflags, flags.p, 4, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hflags & kFlagBadTree) {
        *mesh_error = true;
        *msg = "LBVH construction produced a malformed hierarchy";
        return cudaSuccess;
    }
    if (hflags & kFlagBadVertex) {
        *mesh_error = true;
        *msg = "an instance map is singular or its inverse is not finite";
        return cudaSuccess;
    }
    S.built = true;
    S.bvh_ready = !S.two_level;
    S.tl_ready = S.two_level;
    return cudaSuccess;
}

// ------------------------------------------------------------------ instanced scenes
// Instance i of prototype iproto[i] owns world vertices vbase[i] .. vbase[i+1] and triangles tbase[i] ..
// tbase[i+1]; the instance of an element is found by binary search over the (ascending) bases.
namespace {

__device__ __forceinline__ int instance_of(const int64_t* base, int32_t n_inst, int64_t e) {
    int lo = 0, hi = n_inst - 1;  // largest i with base[i] <= e (base[0] = 0 <= e)
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (base[mid] <= e) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// x' = A x + b per instance, each component ((A_r0 x + A_r1 y) + A_r2 z) + b_r, every product and sum
// rounded to float32 in that order (this unit is compiled without contraction)
__global__ void k_inst_verts(const float* __restrict__ pv, const int64_t* __restrict__ pvoff,
                             const int32_t* __restrict__ iproto, const int64_t* __restrict__ vbase,
                             const float* __restrict__ xf, int32_t n_inst, int64_t nv, float* __restrict__ out) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x) {
        const int i = instance_of(vbase, n_inst, v);
        const int64_t src = pvoff[iproto[i]] + (v - vbase[i]);
        const float x = pv[3 * src], y = pv[3 * src + 1], z = pv[3 * src + 2];
        const float* a = xf + 12 * (int64_t)i;
#pragma unroll
        for (int r = 0; r < 3; ++r)
            out[3 * v + r] = affine_row(make_float4(a[4 * r], a[4 * r + 1], a[4 * r + 2], a[4 * r + 3]), x, y, z);
    }
}

__global__ void k_inst_tris(const int32_t* __restrict__ pt, const int32_t* __restrict__ pmat,
                            const int64_t* __restrict__ ptoff, const int32_t* __restrict__ iproto,
                            const int64_t* __restrict__ vbase, const int64_t* __restrict__ tbase, int32_t n_inst,
                            int64_t nt, int32_t* __restrict__ tris, int32_t* __restrict__ mat,
                            int32_t* __restrict__ obj) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt; t += (int64_t)gridDim.x * blockDim.x) {
        const int i = instance_of(tbase, n_inst, t);
        const int64_t src = ptoff[iproto[i]] + (t - tbase[i]);
        const int32_t off = (int32_t)vbase[i];
#pragma unroll
        for (int k = 0; k < 3; ++k) tris[3 * t + k] = pt[3 * src + k] + off;
        mat[t] = pmat[src];
        obj[t] = i;
    }
}

// Instance records of the two-level structure (8 float4 per instance): rows (A_r, b_r); rows of A^-1 computed
// in float64 and rounded, with |A^-1|_inf rounded up (w of row 0), the prototype's root reference (w of row 1)
// and the first world triangle (w of row 2); the world box of the prototype's vertex bounds pbox under the
// map, from float64 interval arithmetic rounded outwards, grown by the float32 rounding bound of a mapped
// vertex and by pad (w of the box's hi: 1 for a prototype without triangles, which the walk skips).  Also the
// box centre for the top level's Morton keys.  A singular map (or a non-finite inverse) sets kFlagBadVertex.
__global__ void k_inst_records(const float* __restrict__ xf, const int32_t* __restrict__ iproto,
                               const int64_t* __restrict__ tbase, const int64_t* __restrict__ ptoff, int32_t n_inst,
                               const float* __restrict__ pbox, const int32_t* __restrict__ proot, float pad,
                               float4* __restrict__ rec, float* __restrict__ cen, uint32_t* flags) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_inst; i += gridDim.x * blockDim.x) {
        const float* a = xf + 12 * (int64_t)i;
        double A[3][3], b[3];
        for (int r = 0; r < 3; ++r) {
            for (int k = 0; k < 3; ++k) A[r][k] = a[4 * r + k];
            b[r] = a[4 * r + 3];
        }
        const double c00 = A[1][1] * A[2][2] - A[1][2] * A[2][1], c01 = A[1][2] * A[2][0] - A[1][0] * A[2][2],
                     c02 = A[1][0] * A[2][1] - A[1][1] * A[2][0];
        const double det = A[0][0] * c00 + A[0][1] * c01 + A[0][2] * c02;
        double inv[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
        bool ok = isfinite(det) && fabs(det) > 1e-300;
        if (ok) {
            const double id = 1.0 / det;
            inv[0][0] = c00 * id;
            inv[1][0] = c01 * id;
            inv[2][0] = c02 * id;
            inv[0][1] = (A[0][2] * A[2][1] - A[0][1] * A[2][2]) * id;
            inv[1][1] = (A[0][0] * A[2][2] - A[0][2] * A[2][0]) * id;
            inv[2][1] = (A[0][1] * A[2][0] - A[0][0] * A[2][1]) * id;
            inv[0][2] = (A[0][1] * A[1][2] - A[0][2] * A[1][1]) * id;
            inv[1][2] = (A[0][2] * A[1][0] - A[0][0] * A[1][2]) * id;
            inv[2][2] = (A[0][0] * A[1][1] - A[0][1] * A[1][0]) * id;
        }
        float fi[3][3];
        double ninv = 0.0;
        for (int r = 0; r < 3; ++r) {
            double row = 0.0;
            for (int k = 0; k < 3; ++k) {
                fi[r][k] = (float)inv[r][k];
                ok = ok && isfinite(fi[r][k]);
                row += fabs((double)fi[r][k]);
            }
            ninv = fmax(ninv, row);
        }
        if (!ok) atomicOr(flags, kFlagBadVertex);
        const int q = iproto[i];
        const bool empty = ptoff[q + 1] == ptoff[q];
        const float* pb = pbox + 6 * q;
        float lo[3], hi[3];
        for (int r = 0; r < 3; ++r) {
            double c = b[r], e = 0.0, mag = fabs(b[r]);
            for (int k = 0; k < 3; ++k) {
                const double l = pb[k], h = pb[3 + k];
                c += A[r][k] * (0.5 * (l + h));
                e += fabs(A[r][k]) * (0.5 * (h - l));
                mag += fabs(A[r][k]) * fmax(fabs(l), fabs(h));
            }
            const double slack = mag * 4.76837158203125e-07;  // 2^-21: six float32 roundings of the mapped vertex
            lo[r] = __fsub_rd(__double2float_rd(c - e - slack), pad);
            hi[r] = __fadd_ru(__double2float_ru(c + e + slack), pad);
        }
        float4* o = rec + 8 * (int64_t)i;
        for (int r = 0; r < 3; ++r) o[r] = make_float4(a[4 * r], a[4 * r + 1], a[4 * r + 2], a[4 * r + 3]);
        o[3] = make_float4(fi[0][0], fi[0][1], fi[0][2], __double2float_ru(ninv * (1.0 + 1e-6)));
        o[4] = make_float4(fi[1][0], fi[1][1], fi[1][2], __int_as_float(proot[q]));
        o[5] = make_float4(fi[2][0], fi[2][1], fi[2][2], __int_as_float((int32_t)tbase[i]));
        o[6] = make_float4(lo[0], lo[1], lo[2], 0.0f);
        o[7] = make_float4(hi[0], hi[1], hi[2], empty ? 1.0f : 0.0f);
        for (int r = 0; r < 3; ++r) cen[3 * (int64_t)i + r] = 0.5f * lo[r] + 0.5f * hi[r];
    }
}

// Tighter world boxes: the bounds of each instance's expanded world vertices (the very vertices its
// triangles are tested with) grown by pad, intersected with the box from the map; one warp per instance.
__global__ void k_inst_world_boxes(const float* __restrict__ V, const int64_t* __restrict__ vbase, int32_t n_inst,
                                   float pad, float4* __restrict__ rec, float* __restrict__ cen) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n_inst; i += warps) {
        float lo[3] = {3.0e38f, 3.0e38f, 3.0e38f}, hi[3] = {-3.0e38f, -3.0e38f, -3.0e38f};
        for (int64_t v = vbase[i] + lane; v < vbase[i + 1]; v += 32)
            for (int k = 0; k < 3; ++k) {
                lo[k] = fminf(lo[k], V[3 * v + k]);
                hi[k] = fmaxf(hi[k], V[3 * v + k]);
            }
        for (int o = 16; o > 0; o >>= 1)
            for (int k = 0; k < 3; ++k) {
                lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
                hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
            }
        if (lane == 0 && vbase[i + 1] > vbase[i]) {
            float4* o = rec + 8 * i;
            const float4 l0 = o[6], h0 = o[7];
            const float4 l = make_float4(fmaxf(l0.x, __fsub_rd(lo[0], pad)), fmaxf(l0.y, __fsub_rd(lo[1], pad)),
                                         fmaxf(l0.z, __fsub_rd(lo[2], pad)), 0.0f);
            const float4 h = make_float4(fminf(h0.x, __fadd_ru(hi[0], pad)), fminf(h0.y, __fadd_ru(hi[1], pad)),
                                         fminf(h0.z, __fadd_ru(hi[2], pad)), h0.w);
            o[6] = l;
            o[7] = h;
            cen[3 * i] = 0.5f * l.x + 0.5f * h.x;
            cen[3 * i + 1] = 0.5f * l.y + 0.5f * h.y;
            cen[3 * i + 2] = 0.5f * l.z + 0.5f * h.z;
        }
    }
}

// top level of at most kLeafMax instances: one root node holding each instance as a leaf of its own
__global__ void k_tlas_small(const float4* __restrict__ rec, const int32_t* __restrict__ tinst, int32_t n,
                             float4* __restrict__ nodes) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    float lo[3][4], hi[3][4];
    int32_t ref[4];
    for (int j = 0; j < 4; ++j) {
        const bool use = j < n;
        const float4 l = use ? rec[8 * (int64_t)tinst[j] + 6] : make_float4(0, 0, 0, 0);
        const float4 h = use ? rec[8 * (int64_t)tinst[j] + 7] : make_float4(0, 0, 0, 0);
        lo[0][j] = l.x, lo[1][j] = l.y, lo[2][j] = l.z;
        hi[0][j] = h.x, hi[1][j] = h.y, hi[2][j] = h.z;
        ref[j] = use ? leaf_ref(j, 1) : kEmptyRef;
    }
    for (int k = 0; k < 3; ++k) {
        nodes[2 * k] = make_float4(lo[k][0], lo[k][1], lo[k][2], lo[k][3]);
        nodes[2 * k + 1] = make_float4(hi[k][0], hi[k][1], hi[k][2], hi[k][3]);
    }
    nodes[6] = make_float4(__int_as_float(ref[0]), __int_as_float(ref[1]), __int_as_float(ref[2]),
                           __int_as_float(ref[3]));
    nodes[7] = make_float4(__int_as_float(-1), 0.0f, 0.0f, 0.0f);
}

}  // namespace

// Scratch of one 4-wide build over n primitives (binary topology, boxes, wide-node numbering).
struct WideScratch {
    DevBuf child, range, par_i, par_l, boxes, visits, wflag, widx, wscan, wtotal;
    ~WideScratch() {
        for (DevBuf* b : {&child, &range, &par_i, &par_l, &boxes, &visits, &wflag, &widx, &wscan, &wtotal}) release(*b);
    }
};

// 4-wide BVH over n > kLeafMax primitives whose Morton keys are sorted in keys (leaf p's box from leaf(p)):
// Karras topology, boxes bottom-up, the wide nodes written from nodes[node_off] on (at most node_cap nodes
// in all) with references offset by node_off and leaf codes by leaf_off; the node count in *n4.
template <class LeafBox>
static cudaError_t wide_from_sorted(int n, const uint64_t* keys, LeafBox leaf, float4* nodes, int64_t node_cap,
                                    int32_t node_off, int32_t leaf_off, uint32_t* flags, WideScratch& w,
                                    cudaStream_t s, int64_t* n4_out) {
    CK(grow(w.child, (size_t)(n - 1) * sizeof(int2)));
    CK(grow(w.range, (size_t)(n - 1) * sizeof(int2)));
    CK(grow(w.par_i, (size_t)n * 4));
    CK(grow(w.par_l, (size_t)n * 4));
    CK(grow(w.boxes, (size_t)(n - 1) * 2 * sizeof(Box)));
    CK(grow(w.visits, (size_t)(n - 1) * 4));
    CK(grow(w.wflag, (size_t)(n - 1) * 4));
    CK(grow(w.widx, (size_t)(n - 1) * 4));
    CK(grow(w.wscan, scan_scratch_bytes(n - 1)));
    CK(grow(w.wtotal, 4));
    note_launch();
    k_karras<<<grid_for(n - 1, kB), kB, 0, s>>>(keys, n, ptr<int2>(w.child), ptr<int2>(w.range), ptr<int32_t>(w.par_i),
                                                ptr<int32_t>(w.par_l));
    CK(cudaGetLastError());
    CK(cudaMemsetAsync(w.visits.p, 0, (size_t)(n - 1) * 4, s));
    note_launch();
    k_boxes<<<grid_for(n, kB), kB, 0, s>>>(leaf, n, ptr<int2>(w.child), ptr<int32_t>(w.par_i), ptr<int32_t>(w.par_l),
                                           ptr<Box>(w.boxes), ptr<uint32_t>(w.visits), flags);
    CK(cudaGetLastError());
    note_launch();
    k_wide_flags<<<grid_for(n - 1, kB), kB, 0, s>>>(n, ptr<int2>(w.range), ptr<int32_t>(w.par_i),
                                                    ptr<uint32_t>(w.wflag), flags);
    CK(cudaGetLastError());
    CK(exclusive_scan_u32(ptr<uint32_t>(w.wflag), ptr<uint32_t>(w.widx), n - 1, ptr<uint32_t>(w.wtotal), w.wscan.p, s));
    uint32_t n4 = 0;
    CK(cudaMemcpyAsync(&n4, w.wtotal.p, 4, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if ((int64_t)node_off + n4 > node_cap) return cudaErrorInvalidValue;  // cannot happen: n4 <= n - 1
    note_launch();
    k_pack_wide<<<grid_for(n - 1, kB), kB, 0, s>>>(n, ptr<int2>(w.child), ptr<int2>(w.range), ptr<Box>(w.boxes),
                                                   ptr<uint32_t>(w.wflag), ptr<uint32_t>(w.widx),
                                                   nodes + 8 * (int64_t)node_off, node_off, leaf_off);
    CK(cudaGetLastError());
    *n4_out = n4;
    return cudaSuccess;
}

// The two-level structure of an instanced scene: the prototypes' BVHs (object space, once), then the
// instance records and the top-level BVH over the instances' world boxes (every build and move).
static cudaError_t build_two_level(SceneDev& S, float pad_world, uint32_t* flags, cudaStream_t s) {
    const InstanceDev& I = *S.inst;
    const int32_t P = I.n_proto;
    int64_t nmax = std::max<int64_t>(I.n_inst, 1);
    for (int32_t q = 0; q < P; ++q) nmax = std::max(nmax, I.ptoff_h[q + 1] - I.ptoff_h[q]);
    DevBuf keys, vals, sort_scr, bnd, cen;
    struct Rel {
        DevBuf* b[5];
        ~Rel() {
            for (DevBuf* x : b) release(*x);
        }
    } rel{{&keys, &vals, &sort_scr, &bnd, &cen}};
    CK(grow(keys, (size_t)nmax * 8));
    CK(grow(vals, (size_t)nmax * 4));
    CK(grow(sort_scr, sort_scratch_bytes(nmax)));
    CK(grow(bnd, 64));
    WideScratch w;
    auto bounds = [&](const float* pts, int64_t n, float lo[3], float hi[3]) -> cudaError_t {
        const uint32_t init[6] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u};
        CK(cudaMemcpyAsync(bnd.p, init, sizeof(init), cudaMemcpyHostToDevice, s));
        note_launch();
        k_bounds<<<grid_for(n, kB, 152 * 4), kB, 0, s>>>(pts, n, ptr<uint32_t>(bnd));
        CK(cudaGetLastError());
        uint32_t hb[6];
        CK(cudaMemcpyAsync(hb, bnd.p, sizeof(hb), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        for (int k = 0; k < 6; ++k) {
            const uint32_t u = hb[k], bits = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
            float f;
            memcpy(&f, &bits, 4);
            (k < 3 ? lo[k] : hi[k - 3]) = f;
        }
        return cudaSuccess;
    };
    if (!S.blas_ready) {
        int64_t cap = 1;
        for (int32_t q = 0; q < P; ++q) cap += std::max<int64_t>(I.ptoff_h[q + 1] - I.ptoff_h[q] - 1, 0);
        const int64_t pt = I.ptoff_h[P];
        CK(grow(S.blas_nodes, (size_t)cap * 8 * sizeof(float4)));
        CK(grow(S.blas_tri, (size_t)std::max<int64_t>(pt, 1) * 3 * sizeof(float4)));
        std::vector<int32_t> root(P, kEmptyRef);
        std::vector<float> box(6 * (size_t)P, 0.0f);
        int64_t node_off = 0;
        for (int32_t q = 0; q < P; ++q) {
            const int64_t nvq = I.pvoff_h[q + 1] - I.pvoff_h[q], ntq = I.ptoff_h[q + 1] - I.ptoff_h[q];
            if (ntq == 0 || nvq == 0) continue;
            const float* Vq = ptr<float>(I.pverts) + 3 * I.pvoff_h[q];
            const int32_t* Tq = ptr<int32_t>(I.ptris) + 3 * I.ptoff_h[q];
            float lo[3], hi[3];
            CK(bounds(Vq, nvq, lo, hi));
            double diag2 = 0.0;
            for (int k = 0; k < 3; ++k) {
                box[6 * q + k] = lo[k];
                box[6 * q + 3 + k] = hi[k];
                diag2 += ((double)hi[k] - lo[k]) * ((double)hi[k] - lo[k]);
            }
            const float pad_q = (float)(1e-5 * sqrt(diag2) + 1e-7);
            note_launch();
            k_morton<<<grid_for(ntq, kB), kB, 0, s>>>(Vq, Tq, ntq, ptr<uint32_t>(bnd), ptr<uint64_t>(keys),
                                                      ptr<uint32_t>(vals));
            CK(cudaGetLastError());
            CK(radix_sort_u64(ptr<uint64_t>(keys), ptr<uint32_t>(vals), ntq, 48, sort_scr.p, s));
            note_launch();
            k_reorder<<<grid_for(ntq, kB), kB, 0, s>>>(Vq, Tq, ntq, ptr<uint32_t>(vals),
                                                       ptr<float4>(S.blas_tri) + 3 * I.ptoff_h[q]);
            CK(cudaGetLastError());
            if (ntq <= kLeafMax) {
                root[q] = leaf_ref((int)I.ptoff_h[q], (int)ntq);
            } else {
                int64_t n4 = 0;
                CK(wide_from_sorted((int)ntq, ptr<uint64_t>(keys), TriLeafBox{Vq, Tq, ptr<uint32_t>(vals), pad_q},
                                    ptr<float4>(S.blas_nodes), cap, (int32_t)node_off, (int32_t)I.ptoff_h[q], flags, w,
                                    s, &n4));
                root[q] = (int32_t)node_off;
                node_off += n4;
            }
        }
        S.blas_n_nodes = node_off;
        CK(grow(S.blas_root, (size_t)P * 4));
        CK(grow(S.proto_box, (size_t)P * 24));
        CK(cudaMemcpyAsync(S.blas_root.p, root.data(), (size_t)P * 4, cudaMemcpyHostToDevice, s));
        CK(cudaMemcpyAsync(S.proto_box.p, box.data(), (size_t)P * 24, cudaMemcpyHostToDevice, s));
        CK(cudaStreamSynchronize(s));  // the host tables above go out of scope
        S.blas_ready = true;
    }
    // instance records and the top level
    const int32_t n = I.n_inst;
    CK(grow(S.inst_rec, (size_t)n * 8 * sizeof(float4)));
    CK(grow(S.tlas_inst, (size_t)n * 4));
    CK(grow(cen, (size_t)n * 12));
    note_launch();
    k_inst_records<<<grid_for(n, kB), kB, 0, s>>>(ptr<float>(I.xform), ptr<int32_t>(I.iproto), ptr<int64_t>(I.tbase),
                                                  ptr<int64_t>(I.ptoff), n, ptr<float>(S.proto_box),
                                                  ptr<int32_t>(S.blas_root), pad_world, ptr<float4>(S.inst_rec),
                                                  ptr<float>(cen), flags);
    CK(cudaGetLastError());
    note_launch();
    k_inst_world_boxes<<<grid_for((int64_t)n * 32, kB), kB, 0, s>>>(ptr<float>(S.verts), ptr<int64_t>(I.vbase), n,
                                                                     pad_world, ptr<float4>(S.inst_rec), ptr<float>(cen));
    CK(cudaGetLastError());
    float lo[3], hi[3];
    CK(bounds(ptr<float>(cen), n, lo, hi));
    note_launch();
    k_morton_pts<<<grid_for(n, kB), kB, 0, s>>>(ptr<float>(cen), n, ptr<uint32_t>(bnd), ptr<uint64_t>(keys),
                                                ptr<uint32_t>(vals));
    CK(cudaGetLastError());
    CK(radix_sort_u64(ptr<uint64_t>(keys), ptr<uint32_t>(vals), n, 63, sort_scr.p, s));
    CK(cudaMemcpyAsync(S.tlas_inst.p, vals.p, (size_t)n * 4, cudaMemcpyDeviceToDevice, s));
    if (n <= kLeafMax) {
        if (S.nodes.cap > ((size_t)1 << 20)) release(S.nodes);
        CK(grow(S.nodes, 8 * sizeof(float4)));
        note_launch();
        k_tlas_small<<<1, 32, 0, s>>>(ptr<float4>(S.inst_rec), ptr<int32_t>(S.tlas_inst), n, ptr<float4>(S.nodes));
        CK(cudaGetLastError());
        S.n_nodes = 1;
    } else {
        const size_t need = (size_t)(n - 1) * 8 * sizeof(float4);
        if (S.nodes.cap > 4 * need + ((size_t)1 << 20)) release(S.nodes);  // a flat scene's hierarchy before
        CK(grow(S.nodes, need));
        int64_t n4 = 0;
        CK(wide_from_sorted(n, ptr<uint64_t>(keys), InstLeafBox{ptr<float4>(S.inst_rec), ptr<int32_t>(S.tlas_inst)},
                            ptr<float4>(S.nodes), n - 1, 0, 0, flags, w, s, &n4));
        S.n_nodes = n4;
    }
    S.root = 0;
    return cudaSuccess;
}

cudaError_t expand_instance_verts(const InstanceDev& I, const float* xf, float* out, cudaStream_t s) {
    if (I.nv == 0) return cudaSuccess;
    note_launch();
    k_inst_verts<<<grid_for(I.nv, kB), kB, 0, s>>>(ptr<float>(I.pverts), ptr<int64_t>(I.pvoff), ptr<int32_t>(I.iproto),
                                                   ptr<int64_t>(I.vbase), xf, I.n_inst, I.nv, out);
    return cudaGetLastError();
}

cudaError_t expand_instance_tris(const InstanceDev& I, int32_t* tris, int32_t* mat, int32_t* obj, cudaStream_t s) {
    if (I.nt == 0) return cudaSuccess;
    note_launch();
    k_inst_tris<<<grid_for(I.nt, kB), kB, 0, s>>>(ptr<int32_t>(I.ptris), ptr<int32_t>(I.pmat), ptr<int64_t>(I.ptoff),
                                                  ptr<int32_t>(I.iproto), ptr<int64_t>(I.vbase), ptr<int64_t>(I.tbase),
                                                  I.n_inst, I.nt, tris, mat, obj);
    return cudaGetLastError();
}

}  // namespace st
