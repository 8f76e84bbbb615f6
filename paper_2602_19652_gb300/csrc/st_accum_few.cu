// Spectrum accumulation (Eq. 2-4 specular, Eq. 7-8 diffraction) for few frequency bins or few microphones,
// omnidirectional receivers (the paper's setups: 32 and 64 microphones x 14 bins).
//
// The general accumulator gives a thread 16 bins of a microphone pair; with 14 bins its CTA is one thread per pair -- 16
// threads for 32 microphones -- that form the anchors, the per-(path, bin) factors and the terms in turn, and thousands of
// such CTAs leave as many partial spectra to sum.  Here a CTA of 256 threads is PG path groups x TM microphones x NS runs
// of at most KT bins: the groups consume different paths of the tile, and all threads share the anchors, which at this
// size are most of the work (about 300 instructions a (path, microphone), 100-150 for its 14 terms).  Bound by issue;
// what it measures: 64 microphones x 14 bins, 377k specular and 835k diffraction paths, 2.30 -> 1.37 ms; 32 x 14, 42k and
// 185k paths, 0.32 -> 0.14 ms; 4 x 14, 104k and 185k, 0.54 -> 0.055 ms.  (Small arrays over a few hundred bins gain
// likewise: the general tile's per-(path, bin) factors serve only their few pairs.)
//
// A thread owns one run of one microphone, its even and odd bins as the two halves of packed registers.  Per tile, while
// the previous one is consumed (one barrier a tile): per (path, bin) log2 of the reflection product (or the diffraction
// factor) and the emitter's directivity, four bins a thread; per (path, microphone) r = r_pre + |m - P| in float-float,
// gamma^2, the phasor at each run's first bin and the one-bin step.  The path groups' sums are added in group order and
// the chunks' partial spectra afterwards (fixed order, no float atomics).  Shared-memory pointers are the CTA's base plus
// an integer offset: rounding a pointer up through an integer makes the compiler use generic loads and 64-bit indices.
#include <math.h>

#include <algorithm>

#include "st_accum_dev.cuh"
#include "st_internal.cuh"

namespace st {

namespace {

using namespace acc;

constexpr int kFewThreads = 256;

struct FewGeom {
    int KT, TM, NS, PG, PT;  // bins per run, microphones, runs, path groups, paths per tile (a multiple of PG)
    int n_mb;                // microphone blocks
    int cached, direct;      // material rows in shared memory; diffraction factors read from them in place
    int buf_bytes, smem;
};

__host__ __device__ constexpr int few_stride(int kt) {  // floats of a run's row: 128-bit rows, 4 mod 8 (no conflicts)
    const int s = (kt + 3) & ~3;
    return (s & 4) ? s : s + 4;
}

struct FewBuf {
    float2* z;  // [PT][NS][TM] phasor at the run's first bin
    float2* w;  // [PT][TM] one-bin step
    float* ng;  // [PT][TM] -gamma^2
    float* x;   // [PT][NS][stride] log2 of the factors
    int* mat;   // [PT] material of the last hit, -1: no path
};

__device__ __forceinline__ FewBuf few_buf(char* base, const FewGeom& g, int b) {
    const int nw = g.PT * g.TM, st = few_stride(g.KT);
    int o = b * g.buf_bytes;
    FewBuf B;
    B.z = reinterpret_cast<float2*>(base + o);
    o += nw * g.NS * 8;
    B.w = reinterpret_cast<float2*>(base + o);
    o += nw * 8;
    B.ng = reinterpret_cast<float*>(base + o);
    o = (o + nw * 4 + 15) & ~15;
    B.x = reinterpret_cast<float*>(base + o);
    o += g.direct ? 0 : g.PT * g.NS * st * 4;
    B.mat = reinterpret_cast<int*>(base + o);
    return B;
}

// log2 of the factors of bins 4 v .. 4 v + 3 of run s, path data d
template <int KIND>
__device__ __forceinline__ float4 few_factors(const AccumArgs& a, const FewGeom& g, const float* d, const float* mt,
                                              int s, int v) {
    const int st = few_stride(g.KT);
    const float4 dd = *reinterpret_cast<const float4*>(d + 8);  // meta, chain, emitter coordinate
    const uint32_t meta = __float_as_uint(dd.x), c0 = __float_as_uint(dd.y), c1 = __float_as_uint(dd.z);
    const int matj = (meta >> 8) & 255, k = s * g.KT + 4 * v, n = min(g.KT - 4 * v, a.F - k);
    auto row = [&](int mq) -> float4 {
        if (g.cached) return *reinterpret_cast<const float4*>(mt + (mq * g.NS + s) * st + 4 * v);
        const float* t = (KIND == 1 ? a.lid : a.lk) + (int64_t)mq * a.F + k;
        return make_float4(n > 0 ? t[0] : kNegInf, n > 1 ? t[1] : kNegInf, n > 2 ? t[2] : kNegInf,
                           n > 3 ? t[3] : kNegInf);
    };
    float4 x;
    if (KIND == 1 || a.reflection_mode == 1) {
        x = row(matj);
    } else {
        const int len = meta & 15;
        x = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < len; ++q) {
            const float4 r = row((q < 4 ? (c0 >> (8 * q)) : (c1 >> (8 * (q - 4)))) & 255);
            x = make_float4(x.x + r.x, x.y + r.y, x.z + r.z, x.w + r.w);
        }
    }
    if (a.etab && dd.w >= 0.0f) {  // emitter directivity, linear between the table's rows
        const int it = min((int)dd.w, a.n_theta - 2);
        const float w = dd.w - (float)it;
        const float* e0 = a.etab + (int64_t)it * a.F + k;
        const float* e1 = e0 + a.F;
        float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < n) {
                const float de = (1.0f - w) * e0[c] + w * e1[c];
                xs[c] += de > 0.0f ? log2f(de) : kNegInf;
            }
        x = make_float4(xs[0], xs[1], xs[2], xs[3]);
    }
    return x;
}

// factors and anchors of one tile of np paths (reads pd, writes buffer B)
template <int KIND>
__device__ __forceinline__ void few_produce(const AccumArgs& a, const FewGeom& g, const FewBuf& B, const float* pd, int np,
                                            const float* mt, const float* mics, int mic0, int64_t pglob) {
    const int PT = g.PT, NS = g.NS, TM = g.TM, tid = threadIdx.x, nthr = blockDim.x;
    for (int p = tid; p < PT; p += nthr) B.mat[p] = p < np ? (int)((__float_as_uint(pd[p * 12 + 8]) >> 8) & 255u) : -1;
    if (!g.direct) {
        const int st = few_stride(g.KT), nv = (g.KT + 3) >> 2, per = NS * nv;
        const float inv_per = 1.0f / (float)per, inv_nv = 1.0f / (float)nv;
        for (int e = tid; e < np * per; e += nthr) {
            const int p = __float2int_rz(((float)e + 0.5f) * inv_per), i = e - p * per;
            const int s = __float2int_rz(((float)i + 0.5f) * inv_nv), v = i - s * nv;
            *reinterpret_cast<float4*>(B.x + (p * NS + s) * st + 4 * v) = few_factors<KIND>(a, g, pd + p * 12, mt, s, v);
        }
    }
    const float inv_tm = 1.0f / (float)TM;
    for (int e = tid; e < PT * TM; e += nthr) {
        const int p = __float2int_rz(((float)e + 0.5f) * inv_tm), ml = e - p * TM, m = mic0 + ml;
        float2* zo = B.z + p * NS * TM + ml;
        // (per-microphone receiver test: a microphone that does not see the path gets a zero anchor)
        if (p >= np || m >= a.M || (a.mask && !((a.mask[pglob + p] >> m) & 1ull))) {
            for (int s = 0; s < NS; ++s) zo[s * TM] = make_float2(0.0f, 0.0f);
            B.w[e] = make_float2(0.0f, 0.0f);
            if (KIND == 0) B.ng[e] = 0.0f;
            continue;
        }
        const float* d = pd + p * 12;
        const float mx = mics[3 * ml], my = mics[3 * ml + 1], mz = mics[3 * ml + 2];
        float inv;
        const ff dist = dist_inv_ff(mx, my, mz, d[0], d[1], d[2], &inv);
        const ff r = ff_add(ff{d[6], d[7]}, dist);
        const float rh = r.hi, ir = rcp(rh);
        if (KIND == 0) {
            const float ux = (mx - d[0]) * inv, uy = (my - d[1]) * inv, uz = (mz - d[2]) * inv;
            const float cg = d[3] * ux + d[4] * uy + d[5] * uz;
            const float cx = d[4] * uz - d[5] * uy, cy = d[5] * ux - d[3] * uz, cz = d[3] * uy - d[4] * ux;
            const float gm = atan2f(sqrtf(cx * cx + cy * cy + cz * cz), cg);
            B.ng[e] = -(gm * gm);
        }
        float sn, cs;
        sincospif(2.0f * ff_frac(ff_mul(r, ff{a.qhi[0], a.qlo[0]})), &sn, &cs);
        const float A = ir * ir * ex2(rh * a.atm2_0);
        float2 z = make_float2(A * cs, A * sn);
        sincospif(2.0f * ff_frac(ff_mul(r, ff{a.dq_hi, a.dq_lo})), &sn, &cs);
        const float a1 = ex2(rh * a.atm2_step);
        const float2 w1 = make_float2(a1 * cs, a1 * sn);
        B.w[e] = w1;
        *zo = z;
        if (NS > 1) {  // the step between runs, W^KT by its binary digits
            float2 wk = make_float2(1.0f, 0.0f), b = w1;
            for (int n = g.KT;;) {
                if (n & 1) wk = cmul(wk, b);
                if ((n >>= 1) == 0) break;
                b = cmul(b, b);
            }
            for (int s = 1; s < NS; ++s) {
                z = cmul(z, wk);
                zo[s * TM] = z;
            }
        }
    }
}

template <int KT, int KIND>
__global__ void __launch_bounds__(kFewThreads, 3) k_accum_few(const AccumArgs a, const FewGeom g) {
    static_assert(KT % 2 == 0, "bins go in pairs");
    extern __shared__ float4 smem4[];
    char* base = reinterpret_cast<char*>(smem4);
    constexpr int ST = few_stride(KT), NV = (KT + 3) / 4, KP = KT / 2;
    const int PT = g.PT, NS = g.NS, TM = g.TM, PG = g.PG, TN = TM * NS;
    int o = 2 * g.buf_bytes;
    float* pdb = reinterpret_cast<float*>(base + o);  // [2][PT][12]
    o += 2 * PT * 48;
    int* pvb = reinterpret_cast<int*>(base + o);  // [2][PT]
    o += 2 * PT * 4;
    float* mics = reinterpret_cast<float*>(base + o);  // [TM][3]
    o = (o + TM * 12 + 15) & ~15;
    float* mt = reinterpret_cast<float*>(base + o);  // log2 factor rows of the materials, then (specular) g rows
    const int rows = g.cached ? a.n_mat_tab * NS * ST : 0;
    const float* mg = mt + rows;

    const int mic0 = (int)blockIdx.x * TM, by = blockIdx.y;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int grp = tid / TN, tn = tid - grp * TN, tm = tn % TM, s = tn / TM;
    const int k0 = s * KT, kn = min(KT, a.F - k0);  // this thread's bins

    const int64_t pb0 = a.d_base ? (int64_t)*a.d_base : 0;
    const int64_t count = (int64_t)*a.d_count;
    const int64_t n_tiles = (count + PT - 1) / PT;
    const int64_t per = (n_tiles + a.n_chunks - 1) / a.n_chunks;
    const int64_t t0 = (int64_t)by * per, t1 = min(n_tiles, t0 + per);

    u64 Sr[KP], Si[KP];  // even and odd bins
#pragma unroll
    for (int k = 0; k < KP; ++k) Sr[k] = Si[k] = 0ull;

    if (t0 < t1) {
        for (int i = tid; i < 3 * TM; i += nthr) mics[i] = mic0 + i / 3 < a.M ? a.mics[3 * mic0 + i] : 0.0f;
        for (int e = tid; e < rows; e += nthr) {
            const int row = e / ST, kk = e - row * ST, mat = row / NS, k = (row - mat * NS) * KT + kk;
            const bool in = kk < KT && k < a.F;
            const int64_t src = (int64_t)mat * a.F + k;
            mt[e] = in ? (KIND == 1 ? a.lid[src] : a.lk[src]) : kNegInf;
            if (KIND == 0) mt[rows + e] = in ? a.g2[src] : 0.0f;
        }
        load_paths<KIND>(a, PT, t0 * PT, count, pdb, pvb);
        if (t0 + 1 < t1) load_paths<KIND>(a, PT, (t0 + 1) * PT, count, pdb + PT * 12, pvb + PT);
        __syncthreads();
        few_produce<KIND>(a, g, few_buf(base, g, 0), pdb, (int)min((int64_t)PT, count - t0 * PT), mt, mics, mic0,
                          pb0 + t0 * PT);
        __syncthreads();
    }
    for (int64_t tile = t0; tile < t1; ++tile) {
        const int b = (int)((tile - t0) & 1);
        // path data of tile + 2, in flight during this tile (its place was read by the producer a tile ago)
        if (tile + 2 < t1) load_paths_async<KIND>(a, PT, (tile + 2) * PT, count, pdb + b * PT * 12, pvb + b * PT);
        if (tile + 1 < t1) {
            const int nb = b ^ 1;
            few_produce<KIND>(a, g, few_buf(base, g, nb), pdb + nb * PT * 12, (int)min((int64_t)PT, count - (tile + 1) * PT),
                              mt, mics, mic0, pb0 + (tile + 1) * PT);
        }
        const FewBuf C = few_buf(base, g, b);
        for (int p = grp; p < PT; p += PG) {
            const int mat = C.mat[p];
            if (mat < 0) break;  // only the list's last tile has places without a path, at its end
            const float2 z = C.z[(p * NS + s) * TM + tm], w = C.w[p * TM + tm];
            const float n = KIND == 0 ? C.ng[p * TM + tm] : 0.0f;
            // even bins from z, odd bins from z W, both stepping by W^2
            const float2 zo = cmul(z, w), w2 = cmul(w, w);
            u64 zr = pk2(z.x, zo.x), zi = pk2(z.y, zo.y);
            const u64 w2r = pk2(w2.x, w2.x), w2i = pk2(w2.y, w2.y), nw2i = pk2(-w2.y, -w2.y), n2 = pk2(n, n);
            const ulonglong2* xrow =
                reinterpret_cast<const ulonglong2*>(g.direct ? mt + (mat * NS + s) * ST : C.x + (p * NS + s) * ST);
            const ulonglong2* grow = reinterpret_cast<const ulonglong2*>(mg + (mat * NS + s) * ST);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const ulonglong2 x = xrow[v];
                u64 xs[2] = {x.x, x.y};
                if (KIND == 0) {
                    u64 gs[2];
                    if (g.cached) {
                        const ulonglong2 gv = grow[v];
                        gs[0] = gv.x;
                        gs[1] = gv.y;
                    } else {
                        const float* t = a.g2 + (int64_t)mat * a.F + k0 + 4 * v;
                        const int left = kn - 4 * v;
                        gs[0] = pk2(left > 0 ? t[0] : 0.f, left > 1 ? t[1] : 0.f);
                        gs[1] = pk2(left > 2 ? t[2] : 0.f, left > 3 ? t[3] : 0.f);
                    }
                    xs[0] = ffma2(n2, gs[0], xs[0]);
                    xs[1] = ffma2(n2, gs[1], xs[1]);
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int j = 2 * v + c;
                    if (j >= KP) continue;
                    const float2 y = up2(xs[c]);
                    const u64 E = pk2(ex2(y.x), ex2(y.y));
                    Sr[j] = ffma2(E, zr, Sr[j]);
                    Si[j] = ffma2(E, zi, Si[j]);
                    if (j + 1 < KP) cmul2(zr, zi, w2r, w2i, nw2i);
                }
            }
        }
        cp_async_wait_all();
        __syncthreads();
    }
    // ---- partial spectra of this chunk: the path groups' sums in group order, two bin pairs of every run a pass
    float4* red = reinterpret_cast<float4*>(base);  // [2][PG][TN] (re, re, im, im) of a bin pair
#pragma unroll
    for (int v = 0; v < (KP + 1) / 2; ++v) {
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int j = 2 * v + c;
            if (j < KP) {
                const float2 re = up2(Sr[j]), im = up2(Si[j]);
                red[(c * PG + grp) * TN + tn] = make_float4(re.x, re.y, im.x, im.y);
            }
        }
        __syncthreads();
        for (int e = tid; e < 2 * TN; e += nthr) {
            const int c = e / TN, t = e - c * TN, kk = 2 * (2 * v + c), k = t / TM * KT + kk, m = mic0 + t % TM;
            if (kk >= KT || k >= a.F || m >= a.M) continue;
            float4 acc = red[c * PG * TN + t];
            for (int q = 1; q < PG; ++q) {
                const float4 u = red[(c * PG + q) * TN + t];
                acc.x += u.x;
                acc.y += u.y;
                acc.z += u.z;
                acc.w += u.w;
            }
            float2* out = a.partial + ((size_t)by * a.M + m) * a.F + k;
            out[0] = make_float2(acc.x, acc.z);
            if (k + 1 < a.F) out[1] = make_float2(acc.y, acc.w);
        }
    }
}

FewGeom few_geom(const AccumArgs& a) {
    FewGeom g{};
    // run length with the fewest slots over all bins
    int slots = 1 << 30;
    for (int kt : {24, 18, 14}) {
        const int n = (a.F + kt - 1) / kt * kt;
        if (n < slots) {
            slots = n;
            g.KT = kt;
        }
    }
    const int st = few_stride(g.KT);
    g.NS = (a.F + g.KT - 1) / g.KT;
    const int tm = std::max(1, std::min({a.M, a.tile_tp > 0 ? 2 * a.tile_tp : 32, 32, kFewThreads / g.NS}));
    g.n_mb = (a.M + tm - 1) / tm;
    g.TM = (a.M + g.n_mb - 1) / g.n_mb;
    g.PG = std::max(1, kFewThreads / (g.TM * g.NS));
    const int rows = a.n_mat_tab * g.NS * st * 4 * (a.kind == 0 ? 2 : 1);
    g.cached = rows <= 40 * 1024 ? 1 : 0;
    // diffraction without an emitter table: the factor is the material's row, read in place
    g.direct = a.kind == 1 && !a.etab && g.cached ? 1 : 0;
    const int per_path = g.TM * (8 * g.NS + 12) + (g.direct ? 0 : g.NS * st * 4) + 4;
    const int fixed = (g.cached ? rows : 0) + g.TM * 12 + 64;
    const int budget = few_budget(a.tile_kb);
    const int most = std::max(1, std::min(128, (budget - fixed) / (2 * per_path + 2 * 52)));
    while (g.PG > most) g.PG = (g.PG + 1) / 2;
    // paths per tile: about two rounds of anchors for the CTA's threads
    const int threads = g.TM * g.NS * g.PG, want = std::max(g.PG, 2 * threads / g.TM);
    g.PT = std::max(g.PG, std::min(most, want) / g.PG * g.PG);
    g.buf_bytes = (per_path * g.PT + 16 + 255) & ~255;
    g.smem = std::max(2 * g.buf_bytes + 2 * g.PT * 52 + fixed, 2 * threads * 16);
    return g;
}

template <int KT, int KIND>
cudaError_t launch_few(const AccumArgs& a, const FewGeom& g, cudaStream_t s) {
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e =
            cudaFuncSetAttribute(k_accum_few<KT, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    dim3 grid((unsigned)g.n_mb, (unsigned)a.n_chunks);
    note_launch();
    k_accum_few<KT, KIND><<<grid, g.TM * g.NS * g.PG, g.smem, s>>>(a, g);
    return cudaGetLastError();
}

template <int KIND>
cudaError_t launch_few_kt(const AccumArgs& a, const FewGeom& g, cudaStream_t s) {
    if (g.KT == 14) return launch_few<14, KIND>(a, g, s);
    return g.KT == 18 ? launch_few<18, KIND>(a, g, s) : launch_few<24, KIND>(a, g, s);
}

}  // namespace

int32_t few_chunks(const AccumArgs& a, int64_t n_paths) {
    const FewGeom g = few_geom(a);
    const int64_t resident = std::max(1, std::min(3, (220 * 1024) / g.smem));
    const int64_t want = std::max<int64_t>(1, 152 * resident / g.n_mb);
    const int64_t tiles = std::max<int64_t>(1, (n_paths + g.PT - 1) / g.PT);
    return (int32_t)std::min(want, tiles);
}

cudaError_t accumulate_few(const AccumArgs& a, cudaStream_t s) {
    const FewGeom g = few_geom(a);
    return a.kind == 0 ? launch_few_kt<0>(a, g, s) : launch_few_kt<1>(a, g, s);
}

}  // namespace st
