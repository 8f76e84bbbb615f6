// Device-wide primitives: stable LSD radix sort of (u32 or u64 key, u32 value) pairs, compaction of flags, and scans.
//
// Radix sort, 8-bit digits, three launches a pass: digit histograms of the tiles; for every digit the exclusive scan of
// its row of tile counts (one block a digit); the scatter.  A warp owns a contiguous stretch of its tile and ranks it
// with match masks against counters of its own (lanes with equal digits by lane, rounds by position), so the block meets
// twice a tile: equal keys keep their input order.  The number of keys may be on the device (tiles past it do nothing).
// Bound by launches and latency for short arrays, by the scattered writes for long ones.  Against the form before (a
// histogram scanned over three launches, a scatter of 16 rounds with three block barriers each, always 64-bit keys and an
// even number of passes over the array's capacity): mesh pre-processing of 200k triangles 3250 -> 2640 us, a frame of 80k
// rays and 500k candidates 970 -> 767 us, a training step in the room 1110 -> 957 us.
#include <algorithm>
#include <utility>

#include "st_internal.cuh"

namespace st {

namespace {

constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsItems = 16, kRsItemsFew = 4;   // keys per thread; the smaller tile spreads short arrays over the GPU
constexpr int64_t kRsFew = 512 * 1024;          // keys up to which the smaller tile is taken (about two tiles an SM)

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <class K, int ITEMS>
__global__ void __launch_bounds__(kRsThreads) k_rs_hist(const K* __restrict__ keys, int64_t n_max,
                                                        const uint32_t* __restrict__ d_n, int shift,
                                                        uint32_t* __restrict__ hist, int nb) {
    __shared__ uint32_t h[256];
    const int tid = threadIdx.x;
    const int64_t n = d_n ? min((int64_t)*d_n, n_max) : n_max;
    h[tid] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (kRsThreads * ITEMS);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = base + (int64_t)r * kRsThreads + tid;
        if (i < n) atomicAdd(&h[(unsigned)(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[(int64_t)tid * nb + blockIdx.x] = h[tid];
}

// inclusive scan over the block of one value per thread (s_w: one word per warp)
__device__ __forceinline__ uint32_t rs_block_incl(uint32_t x, uint32_t* s_w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w)
        if (w < warp) before += s_w[w];
    __syncthreads();
    return x + before;
}

// one block per digit: exclusive scan of its row of tile counts, the row's total
__global__ void __launch_bounds__(kRsThreads) k_rs_rows(uint32_t* hist, int nb, uint32_t* __restrict__ totals) {
    __shared__ uint32_t s_w[kRsWarps], s_last;
    uint32_t* row = hist + (int64_t)blockIdx.x * nb;
    uint32_t carry = 0;
    for (int b0 = 0; b0 < nb; b0 += kRsThreads) {
        const int i = b0 + threadIdx.x;
        const uint32_t v = i < nb ? row[i] : 0u, incl = rs_block_incl(v, s_w);
        if (i < nb) row[i] = carry + incl - v;
        if (threadIdx.x == kRsThreads - 1) s_last = incl;
        __syncthreads();
        carry += s_last;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

template <class K, int ITEMS>
__global__ void __launch_bounds__(kRsThreads) k_rs_scatter(const K* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                           K* __restrict__ kout, uint32_t* __restrict__ vout,
                                                           int64_t n_max, const uint32_t* __restrict__ d_n, int shift,
                                                           const uint32_t* __restrict__ rows, int nb,
                                                           const uint32_t* __restrict__ totals) {
    __shared__ uint32_t cnt[kRsWarps][256];
    __shared__ uint32_t s_w[kRsWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t n = d_n ? min((int64_t)*d_n, n_max) : n_max;
    const int64_t tile = (int64_t)blockIdx.x * (kRsThreads * ITEMS);
    if (tile >= n) return;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) cnt[w][tid] = 0;
    const uint32_t total = totals[tid];
    const uint32_t base = rs_block_incl(total, s_w) - total + rows[(int64_t)tid * nb + blockIdx.x];
    // (the scan's barriers also publish the zeroed counters)
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t first = tile + (int64_t)warp * 32 * ITEMS + lane;
    K key[ITEMS];
    uint16_t rank[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = first + r * 32;
        const bool valid = i < n;
        key[r] = valid ? kin[i] : (K)0;
        const int d = valid ? (int)((key[r] >> shift) & 255u) : 256;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = valid ? cnt[warp][d] : 0u;
        rank[r] = (uint16_t)(before + __popc(peers & lt_mask));
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) cnt[warp][d] = before + (uint32_t)__popc(peers);
        __syncwarp();
    }
    __syncthreads();
    uint32_t run = base;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) {
        const uint32_t c = cnt[w][tid];
        cnt[w][tid] = run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = first + r * 32;
        if (i < n) {
            const uint32_t pos = cnt[warp][(unsigned)(key[r] >> shift) & 255u] + rank[r];
            kout[pos] = key[r];
            vout[pos] = vin[i];
        }
    }
}

template <class K>
__global__ void k_rs_copy(const K* __restrict__ kin, const uint32_t* __restrict__ vin, K* __restrict__ kout,
                          uint32_t* __restrict__ vout, int64_t n_max, const uint32_t* __restrict__ d_n) {
    const int64_t n = d_n ? min((int64_t)*d_n, n_max) : n_max;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        kout[i] = kin[i];
        vout[i] = vin[i];
    }
}

// ---------------------------------------------------------------- fills
struct FillArgs {
    Fill f[kFillMax];
    int n;
};

__global__ void __launch_bounds__(256) k_fill(const FillArgs a) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    for (int k = 0; k < a.n; ++k) {
        const uint32_t w = a.f[k].word;
        uint32_t* p = static_cast<uint32_t*>(a.f[k].p);
        int64_t words = (int64_t)(a.f[k].bytes / 4);
        // single words up to a 16-byte boundary and after the last one, 128-bit stores between
        const int64_t head = min(words, (int64_t)((16 - (reinterpret_cast<uintptr_t>(p) & 15)) & 15) / 4);
        const int64_t quads = (words - head) / 4;
        uint4* q = reinterpret_cast<uint4*>(p + head);
        for (int64_t i = t; i < quads; i += stride) q[i] = make_uint4(w, w, w, w);
        if (t < head) p[t] = w;
        const int64_t done = head + 4 * quads;
        if (t < words - done) p[done + t] = w;
    }
}

// ---------------------------------------------------------------- compaction of byte flags
constexpr int kCmpThreads = 256, kCmpItems = 16, kCmpTile = kCmpThreads * kCmpItems;

// the thread's 16 flags as a bit mask (non-zero bytes); f is 16-byte aligned
__device__ __forceinline__ uint32_t cmp_mask(const uint8_t* __restrict__ f, int64_t i, int64_t n) {
    uint32_t m = 0;
    if (i + kCmpItems <= n) {
        const uint4 v = *reinterpret_cast<const uint4*>(f + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int b = 0; b < 4; ++b) m |= (uint32_t)(((w[q] >> (8 * b)) & 255u) != 0u) << (4 * q + b);
    } else {
        for (int q = 0; q < kCmpItems; ++q)
            if (i + q < n && f[i + q]) m |= 1u << q;
    }
    return m;
}

__global__ void __launch_bounds__(kCmpThreads) k_cmp_count(const uint8_t* __restrict__ f, int64_t n,
                                                           uint32_t* __restrict__ counts) {
    const int64_t i = (int64_t)blockIdx.x * kCmpTile + (int64_t)threadIdx.x * kCmpItems;
    const uint32_t c = (uint32_t)__popc(cmp_mask(f, i, n));
    const uint32_t sum = __reduce_add_sync(0xffffffffu, c);
    __shared__ uint32_t s_w[kCmpThreads / 32];
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < kCmpThreads / 32; ++w) t += s_w[w];
        counts[blockIdx.x] = t;
    }
}

// tiles up to which a block adds up the counts of the tiles before it itself: 8192 (34M flags) are 134 MB of reads from L2,
// about 20 us; the sum grows with the square of the flags, so beyond it the counts are scanned first (three launches)
constexpr unsigned kCmpSelf = 8192;

// the flagged indices in order; SCANNED: counts hold the sums of the tiles before each (and *total is written), else the
// tiles' own counts, and the last block writes the total
template <bool SCANNED>
__global__ void __launch_bounds__(kCmpThreads) k_cmp_write(const uint8_t* __restrict__ f, int64_t n,
                                                           const uint32_t* __restrict__ counts, uint32_t* __restrict__ idx,
                                                           uint32_t* __restrict__ total) {
    __shared__ uint32_t s_w[kRsWarps];
    uint32_t before = 0;
    if (SCANNED) {
        if (threadIdx.x == 0) before = counts[blockIdx.x];
    } else {
        for (int b = threadIdx.x; b < (int)blockIdx.x; b += kCmpThreads) before += counts[b];
    }
    const int64_t i = (int64_t)blockIdx.x * kCmpTile + (int64_t)threadIdx.x * kCmpItems;
    uint32_t m = cmp_mask(f, i, n);
    const uint32_t c = (uint32_t)__popc(m);
    const uint32_t incl = rs_block_incl(c, s_w);
    const uint32_t before_incl = rs_block_incl(before, s_w);
    __shared__ uint32_t s_base;
    if (threadIdx.x == kCmpThreads - 1) {
        s_base = before_incl;
        if (!SCANNED && blockIdx.x == gridDim.x - 1) *total = before_incl + incl;
    }
    __syncthreads();
    uint32_t pos = s_base + incl - c;
    for (; m; m &= m - 1) idx[pos++] = (uint32_t)(i + __ffs(m) - 1);
}

// ---------------------------------------------------------------- scan
template <class T>
__device__ T warp_incl(T x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Scans one tile per block (in may equal out); writes the block-local scan (inclusive or exclusive) and the tile total.
template <class T, bool Inclusive>
__global__ void __launch_bounds__(kScanThreads) k_scan_tile(const T* in, T* out, int64_t n, T* sums) {
    __shared__ T s_w[kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)tid * kScanItems;
    T v[kScanItems];
    T acc = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const int64_t i = base + j;
        v[j] = i < n ? in[i] : T(0);
        acc += v[j];
    }
    T incl = warp_incl<T>(acc);
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        T w = lane < kScanThreads / 32 ? s_w[lane] : T(0);
        w = warp_incl<T>(w);
        if (lane < kScanThreads / 32) s_w[lane] = w;
    }
    __syncthreads();
    T run = incl - acc + (warp > 0 ? s_w[warp - 1] : T(0));
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const int64_t i = base + j;
        if (Inclusive) run += v[j];
        if (i < n) out[i] = run;
        if (!Inclusive) run += v[j];
    }
    if (tid == kScanThreads - 1 && sums) sums[blockIdx.x] = s_w[kScanThreads / 32 - 1];
}

template <class T>
__global__ void k_scan_add(T* __restrict__ out, int64_t n, const T* __restrict__ add) {
    const int64_t tile = blockIdx.x;
    if (tile == 0) return;
    const T a = add[tile];
    const int64_t base = tile * kScanTile;
    for (int j = threadIdx.x; j < kScanTile; j += blockDim.x) {
        const int64_t i = base + j;
        if (i < n) out[i] += a;
    }
}

template <class T>
__global__ void k_scan_total(const T* in, const T* scanned, int64_t n, T* total) {
    *total = scanned[n - 1] + in[n - 1];
}

// *total holds the last input (saved before an in-place scan); add the last scanned value.
template <class T>
__global__ void k_scan_total_saved(const T* scanned, int64_t n, T* total) {
    *total += scanned[n - 1];
}

template <class T>
size_t scan_bytes_t(int64_t n) {
    size_t b = 0;
    while (n > 1) {
        n = (n + kScanTile - 1) / kScanTile;
        b += ((size_t)n * sizeof(T) + 255) & ~size_t(255);
    }
    return b + 256;
}

// Exclusive scan at every level (block sums are scanned exclusively, then added).
template <class T, bool Inclusive>
cudaError_t scan_impl(const T* in, T* out, int64_t n, void* scratch, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 1) {
        note_launch();
        k_scan_tile<T, Inclusive><<<1, kScanThreads, 0, s>>>(in, out, n, (T*)nullptr);
        return cudaGetLastError();
    }
    T* sums = static_cast<T*>(scratch);
    char* rest = static_cast<char*>(scratch) + (((size_t)nb * sizeof(T) + 255) & ~size_t(255));
    note_launch();
    k_scan_tile<T, Inclusive><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, sums);
    cudaError_t e = scan_impl<T, false>(sums, sums, nb, rest, s);
    if (e != cudaSuccess) return e;
    note_launch();
    k_scan_add<T><<<(unsigned)nb, kScanThreads, 0, s>>>(out, n, sums);
    return cudaGetLastError();
}

}  // namespace

size_t scan_scratch_bytes(int64_t n) { return scan_bytes_t<uint64_t>(n); }

cudaError_t exclusive_scan_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total, void* scratch,
                               cudaStream_t s) {
    if (n <= 0) {
        if (total) return cudaMemsetAsync(total, 0, sizeof(uint32_t), s);
        return cudaSuccess;
    }
    // `total` needs the last input, which an in-place scan overwrites: keep it first.
    if (in == out && total) {
        cudaError_t e = cudaMemcpyAsync(total, in + n - 1, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return e;
        e = scan_impl<uint32_t, false>(in, out, n, scratch, s);
        if (e != cudaSuccess) return e;
        note_launch();
        k_scan_total_saved<uint32_t><<<1, 1, 0, s>>>(out, n, total);
        return cudaGetLastError();
    }
    cudaError_t e = scan_impl<uint32_t, false>(in, out, n, scratch, s);
    if (e != cudaSuccess || !total) return e;
    note_launch();
    k_scan_total<uint32_t><<<1, 1, 0, s>>>(in, out, n, total);
    return cudaGetLastError();
}

cudaError_t inclusive_scan_u64(const uint64_t* in, uint64_t* out, int64_t n, void* scratch, cudaStream_t s) {
    return scan_impl<uint64_t, true>(in, out, n, scratch, s);
}

cudaError_t fill_many(const Fill* f, int n, cudaStream_t s) {
    FillArgs a{};
    size_t most = 0;
    for (int i = 0; i < n && a.n < kFillMax; ++i)
        if (f[i].bytes > 0) {
            a.f[a.n++] = f[i];
            most = std::max(most, f[i].bytes);
        }
    if (a.n == 0) return cudaSuccess;
    note_launch();
    k_fill<<<grid_for((int64_t)((most + 15) / 16), 256, 152 * 8), 256, 0, s>>>(a);
    return cudaGetLastError();
}

size_t compact_scratch_bytes(int64_t n) {
    const int64_t nb = (n + kCmpTile - 1) / kCmpTile;
    return (((size_t)(nb + 1) * 4 + 255) & ~size_t(255)) + scan_scratch_bytes(nb);
}

cudaError_t compact_flags(const uint8_t* flags, int64_t n, uint32_t* idx, uint32_t* total, void* scratch,
                          cudaStream_t s) {
    if (n <= 0) return cudaMemsetAsync(total, 0, sizeof(uint32_t), s);
    const unsigned nb = (unsigned)((n + kCmpTile - 1) / kCmpTile);
    uint32_t* counts = static_cast<uint32_t*>(scratch);
    note_launch();
    k_cmp_count<<<nb, kCmpThreads, 0, s>>>(flags, n, counts);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const bool scanned = nb > kCmpSelf;
    if (scanned) {
        void* scan = static_cast<char*>(scratch) + (((size_t)(nb + 1) * 4 + 255) & ~size_t(255));
        if ((e = exclusive_scan_u32(counts, counts, nb, total, scan, s)) != cudaSuccess) return e;
    }
    note_launch();
    if (scanned) k_cmp_write<true><<<nb, kCmpThreads, 0, s>>>(flags, n, counts, idx, total);
    else k_cmp_write<false><<<nb, kCmpThreads, 0, s>>>(flags, n, counts, idx, total);
    return cudaGetLastError();
}

size_t sort_scratch_bytes(int64_t n) {
    // tiles of n pairs or of any smaller number (scratch made for the largest array serves the others)
    const int64_t few = n < kRsFew ? n : kRsFew;
    const int64_t nb_few = (few + kRsThreads * kRsItemsFew - 1) / (kRsThreads * kRsItemsFew);
    const int64_t nb_all = (n + kRsThreads * kRsItems - 1) / (kRsThreads * kRsItems);
    const int64_t nb = nb_few > nb_all ? nb_few : nb_all;
    size_t b = ((size_t)n * sizeof(uint64_t) + 255) & ~size_t(255);
    b += ((size_t)n * sizeof(uint32_t) + 255) & ~size_t(255);
    b += (size_t)(nb + 1) * 256 * sizeof(uint32_t);
    return b + 512;
}

namespace {

template <class K, int ITEMS>
cudaError_t radix_sort(K* keys, uint32_t* vals, int64_t n, int lo_bit, int hi_bit, void* scratch, cudaStream_t s,
                       const uint32_t* d_n) {
    const int64_t tile = kRsThreads * ITEMS, nb = (n + tile - 1) / tile;
    char* p = static_cast<char*>(scratch);
    K* kb = reinterpret_cast<K*>(p);
    p += ((size_t)n * sizeof(uint64_t) + 255) & ~size_t(255);
    uint32_t* vb = reinterpret_cast<uint32_t*>(p);
    p += ((size_t)n * sizeof(uint32_t) + 255) & ~size_t(255);
    uint32_t* totals = reinterpret_cast<uint32_t*>(p);
    uint32_t* hist = totals + 256;
    K* ka = keys;
    uint32_t* va = vals;
    cudaError_t e;
    for (int shift = lo_bit; shift < hi_bit; shift += 8) {
        note_launch();
        k_rs_hist<K, ITEMS><<<(unsigned)nb, kRsThreads, 0, s>>>(ka, n, d_n, shift, hist, (int)nb);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        note_launch();
        k_rs_rows<<<256, kRsThreads, 0, s>>>(hist, (int)nb, totals);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        note_launch();
        k_rs_scatter<K, ITEMS><<<(unsigned)nb, kRsThreads, 0, s>>>(ka, va, kb, vb, n, d_n, shift, hist, (int)nb, totals);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    if (ka != keys) {  // an odd number of passes: back into the caller's buffers
        note_launch();
        k_rs_copy<K><<<grid_for(n, 256, 152 * 8), 256, 0, s>>>(ka, va, keys, vals, n, d_n);
        return cudaGetLastError();
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t radix_sort_u64(uint64_t* keys, uint32_t* vals, int64_t n, int bits, void* scratch, cudaStream_t s,
                           const uint32_t* d_n) {
    if (n <= 1 || bits <= 0) return cudaSuccess;
    return n <= kRsFew ? radix_sort<uint64_t, kRsItemsFew>(keys, vals, n, 0, bits, scratch, s, d_n)
                       : radix_sort<uint64_t, kRsItems>(keys, vals, n, 0, bits, scratch, s, d_n);
}

cudaError_t radix_sort_u32(uint32_t* keys, uint32_t* vals, int64_t n, int lo_bit, int hi_bit, void* scratch,
                           cudaStream_t s, const uint32_t* d_n) {
    if (n <= 1 || hi_bit <= lo_bit) return cudaSuccess;
    return n <= kRsFew ? radix_sort<uint32_t, kRsItemsFew>(keys, vals, n, lo_bit, hi_bit, scratch, s, d_n)
                       : radix_sort<uint32_t, kRsItems>(keys, vals, n, lo_bit, hi_bit, scratch, s, d_n);
}

}  // namespace st
