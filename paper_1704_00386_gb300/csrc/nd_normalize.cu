// Edge list -> simple undirected CSR, the input form of Section 2 (a simple
// undirected graph: no self-loop, no repeated edge, every edge seen from both
// endpoints, rows sorted).
//
// Every pair (a, b) with a != b emits its two directed keys (a, b) and (b, a),
// packed as (u << B) | v with B = bits of n - 1.  A stable LSD radix sort
// (8-bit digits) orders the keys; equal neighbours are adjacent after the sort,
// so the CSR is the first copy of every key: col = its low B bits, and row_ptr
// [u] = the first unique key whose row is >= u (a binary search per vertex).
//
// Radix pass, tile of kTile keys per block:
//   k_radix_hist   : 256-bin digit histogram of the tile -> hist[d * tiles + t];
//   scan           : exclusive prefix over (digit, tile) gives every tile's
//                    first output slot per digit (stable: tiles in order);
//   k_radix_scatter: stable rank of each key inside its tile (warps walk their
//                    keys in order, peers with the same digit found by one
//                    ballot per digit bit), keys reordered by digit in shared
//                    memory, then written out as contiguous runs.
// Each pass reads the keys twice and writes them once.  The first pass of
// nd_normalize makes its keys from the pairs as it reads them; self-loops
// travel as keys (a, a) and are dropped with the repeats.
// Measured on 33.5M keys of 40 bits (an R-MAT scale-20 edge list): peers by
// __match_any_sync, at 128 registers and so two blocks per SM, kept a scatter
// at 0.375 ms; one atomic per warp on a common cursor
// kept the key emission at 0.37 ms.
#include "nd_internal.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 16;                   // keys per thread per tile
constexpr int kTile = kThreads * kItems;     // 4096 keys per block
constexpr int kPerWarp = kTile / kWarps;     // 512 keys per warp, in rounds of 32
constexpr int kBins = 256;

__device__ __forceinline__ unsigned digit_of(unsigned long long k, int shift) {
    return (unsigned)(k >> shift) & (kBins - 1);
}

// where a radix pass takes key i from: an array of keys, or the pairs
// (key 2i is (src, dst) of pair i, key 2i + 1 is (dst, src); an id outside
// [0, n) raises *err and gives 0)
struct KeyArray {
    const unsigned long long* __restrict__ keys;
    __device__ __forceinline__ unsigned long long operator()(int64_t i) const { return __ldg(keys + i); }
};
struct PairKeys {
    const int64_t* __restrict__ src;
    const int64_t* __restrict__ dst;
    int64_t n;
    int bits;
    int* err;
    __device__ __forceinline__ unsigned long long operator()(int64_t i) const {
        const int64_t a = __ldg(src + (i >> 1)), b = __ldg(dst + (i >> 1));
        if (a < 0 || a >= n || b < 0 || b >= n) {
            atomicOr(err, 1);
            return 0ull;
        }
        return i & 1 ? ((unsigned long long)b << bits) | (unsigned long long)a
                     : ((unsigned long long)a << bits) | (unsigned long long)b;
    }
};

// 256-bin histogram of one tile's digits: hist[d * tiles + t]
template <typename K>
__global__ void __launch_bounds__(kThreads) k_radix_hist(K keys, int64_t count, int shift, int64_t tiles,
                                                         int64_t* __restrict__ hist) {
    __shared__ unsigned h[kBins];
    for (int i = threadIdx.x; i < kBins; i += kThreads) h[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile;
    if (base + kTile <= count) {
#pragma unroll
        for (int k0 = 0; k0 < kItems; k0 += 8) {
            unsigned d[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) d[k] = digit_of(keys(base + (int64_t)(k0 + k) * kThreads + threadIdx.x), shift);
#pragma unroll
            for (int k = 0; k < 8; ++k) atomicAdd(&h[d[k]], 1u);
        }
    } else {
        for (int64_t i = base + threadIdx.x; i < count; i += kThreads) atomicAdd(&h[digit_of(keys(i), shift)], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < kBins; d += kThreads) hist[(int64_t)d * tiles + blockIdx.x] = h[d];
}

// stable scatter of one tile to its digit slots
constexpr int kSThreads = 512;                 // threads of a scatter block
constexpr int kSWarps = kSThreads / 32;
constexpr int kSPerWarp = kTile / kSWarps;      // 256 keys per warp, in rounds of 32
template <typename K>
__global__ void __launch_bounds__(kSThreads, 3) k_radix_scatter(K keys, unsigned long long* __restrict__ out,
                                                                int64_t count, int shift, int64_t tiles,
                                                                const int64_t* __restrict__ offs) {
    __shared__ uint16_t wcount[kSWarps][kBins];  // keys of each digit per warp; then the warp's first slot in the tile
    __shared__ int64_t dout[kBins];              // output slot of the digit's run, less its first slot in the tile
    __shared__ unsigned wsum[kBins / 32];
    __shared__ unsigned long long stage[kTile];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kSWarps * kBins / 2; i += kSThreads) reinterpret_cast<unsigned*>(&wcount[0][0])[i] = 0;
    const int64_t tbase = (int64_t)blockIdx.x * kTile;
    const int64_t wbase = tbase + (int64_t)w * kSPerWarp;
    // 1. stable rank of every key among the earlier keys of its warp with
    //    the same digit: rounds in order, lanes in order inside a round
    unsigned long long key[kSPerWarp / 32];
    unsigned rank[kSPerWarp / 32];
#pragma unroll
    for (int k = 0; k < kSPerWarp / 32; ++k) {
        const int64_t i = wbase + (int64_t)k * 32 + lane;
        key[k] = i < count ? keys(i) : 0ull;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSPerWarp / 32; ++k) {
        const bool ok = wbase + (int64_t)k * 32 + lane < count;  // padding is never counted, never written
        const unsigned d = digit_of(key[k], shift);
        unsigned peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const unsigned m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
            peers &= (d >> b) & 1u ? m : ~m;
        }
        const unsigned before = __popc(peers & ((1u << lane) - 1u));
        const unsigned run = wcount[w][d];
        rank[k] = run + before;
        __syncwarp();
        if (ok && before == 0) wcount[w][d] = (uint16_t)(run + (unsigned)__popc(peers));  // the lowest peer updates
        __syncwarp();
    }
    __syncthreads();
    // 2. per digit: its start inside the tile (exclusive scan over digits),
    //    and the warps' first slots (in warp order)
    unsigned total = 0, incl = 0;
    const int d0 = threadIdx.x;
    if (d0 < kBins) {
#pragma unroll
        for (int v = 0; v < kSWarps; ++v) total += wcount[v][d0];
        incl = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[w] = incl;
    }
    __syncthreads();
    if (d0 < kBins) {
        unsigned run = incl - total;
        for (int v = 0; v < w; ++v) run += wsum[v];
        dout[d0] = offs[(int64_t)d0 * tiles + blockIdx.x] - run;
#pragma unroll
        for (int v = 0; v < kSWarps; ++v) {
            const unsigned c = wcount[v][d0];
            wcount[v][d0] = (uint16_t)run;
            run += c;
        }
    }
    __syncthreads();
    // 3. reorder the tile by digit in shared memory
#pragma unroll
    for (int k = 0; k < kSPerWarp / 32; ++k)
        if (wbase + (int64_t)k * 32 + lane < count) stage[wcount[w][digit_of(key[k], shift)] + rank[k]] = key[k];
    __syncthreads();
    // 4. write the runs out: consecutive threads, consecutive slots
    const int valid = (int)min((int64_t)kTile, count - tbase);
#pragma unroll 4
    for (int p = threadIdx.x; p < valid; p += kSThreads) {
        const unsigned long long k = stage[p];
        out[dout[digit_of(k, shift)] + p] = k;
    }
}

// Of the sorted keys, the first copy of every key that is no self-loop is an
// entry of the CSR.  first[i / 32] holds a bit per key; the number of entries
// before key i is before[i / 32] plus the bits below it in its word.
__device__ __forceinline__ bool is_entry(const unsigned long long* __restrict__ keys, int64_t i, int bits) {
    const unsigned long long k = keys[i];
    return (k >> bits) != (k & ((1ull << bits) - 1ull)) && (i == 0 || keys[i - 1] != k);
}

// the bits of a tile's keys, and how many are set
__global__ void __launch_bounds__(kThreads) k_entry_bits(const unsigned long long* __restrict__ keys, int64_t count,
                                                         int bits, unsigned* __restrict__ first,
                                                         int64_t* __restrict__ tile_entries) {
    __shared__ unsigned wsum[kWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)w * kPerWarp;
    unsigned c = 0;
#pragma unroll 4
    for (int k = 0; k < kPerWarp / 32; ++k) {
        const int64_t i = base + 32 * k + lane;
        const unsigned m = __ballot_sync(0xffffffffu, i < count && is_entry(keys, i, bits));
        if (lane == 0 && i < count) first[i >> 5] = m;
        c += __popc(m);
    }
    if (lane == 0) wsum[w] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0;
        for (int v = 0; v < kWarps; ++v) t += wsum[v];
        tile_entries[blockIdx.x] = t;
    }
}

// the entries' column ids, compacted, and before[] (tile_first: the scanned
// tile_entries)
__global__ void __launch_bounds__(kThreads) k_write_entries(const unsigned long long* __restrict__ keys, int64_t count,
                                                            int bits, const unsigned* __restrict__ first,
                                                            const int64_t* __restrict__ tile_first,
                                                            int64_t* __restrict__ before, int32_t* __restrict__ col) {
    __shared__ unsigned word[kTile / 32];
    const int lane = threadIdx.x & 31;
    const int64_t tile = (int64_t)blockIdx.x * kTile;
    // exclusive scan of the tile's 128 words by the first four warps
    static_assert(kTile / 32 == 128, "one word per thread of the first four warps");
    __shared__ unsigned wsum[4];
    unsigned m = 0, incl = 0;
    if (threadIdx.x < 128) {
        const int64_t i = tile + 32 * (int64_t)threadIdx.x;
        m = i < count ? first[i >> 5] : 0u;
        incl = __popc(m);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[threadIdx.x >> 5] = incl;
    }
    __syncthreads();
    if (threadIdx.x < 128) {
        unsigned add = 0;
        for (int v = 0; v < (int)(threadIdx.x >> 5); ++v) add += wsum[v];
        const unsigned excl = add + incl - __popc(m);
        word[threadIdx.x] = excl;
        const int64_t i = tile + 32 * (int64_t)threadIdx.x;
        if (i < count) before[i >> 5] = tile_first[blockIdx.x] + excl;
    }
    __syncthreads();
    const unsigned long long vmask = (1ull << bits) - 1ull;
    const int64_t base = tile_first[blockIdx.x];
#pragma unroll 4
    for (int k = 0; k < kItems; ++k) {
        const int p = k * kThreads + threadIdx.x;
        const int64_t i = tile + p;
        if (i >= count) break;
        const unsigned mw = first[i >> 5];
        if ((mw >> lane) & 1u)
            col[base + word[p >> 5] + __popc(mw & ((1u << lane) - 1u))] = (int32_t)(keys[i] & vmask);
    }
}

// row_ptr[u] = entries whose row is < u: those before the first key >= u << bits
__global__ void k_row_ptr(const unsigned long long* __restrict__ keys, int64_t count, int64_t n, int bits,
                          const unsigned* __restrict__ first, const int64_t* __restrict__ before, int64_t nnz,
                          int64_t* __restrict__ row_ptr) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u <= n; u += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long x = (unsigned long long)u << bits;
        int64_t lo = 0, hi = count;
        while (lo < hi) {
            const int64_t mid = lo + ((hi - lo) >> 1);
            if (keys[mid] < x) lo = mid + 1; else hi = mid;
        }
        row_ptr[u] = lo < count ? before[lo >> 5] + __popc(first[lo >> 5] & ((1u << (lo & 31)) - 1u)) : nnz;
    }
}

}  // namespace

int nd_id_bits(int64_t n) {
    int b = 1;
    while (b < 63 && ((int64_t)1 << b) < n) ++b;
    return b;
}

namespace {

// one radix pass over the digit at `shift`: keys -> out
template <typename K>
nd_status radix_pass(const K& keys, unsigned long long* out, int64_t count, int shift, int64_t tiles, int64_t* hist,
                     cudaStream_t st) {
    {
        nd_prof_scope ps("radix_hist", st);
        k_radix_hist<K><<<(unsigned)tiles, kThreads, 0, st>>>(keys, count, shift, tiles, hist);
        ND_CUDA(cudaGetLastError());
    }
    ND_CUDA(cudaMemsetAsync(hist + kBins * tiles, 0, sizeof(int64_t), st));
    ND_TRY(nd_scan_i64(hist, (int64_t)kBins * tiles, st));
    nd_prof_scope ps("radix_scatter", st);
    // three blocks of 42 KB per SM
    ND_CUDA(cudaFuncSetAttribute(k_radix_scatter<K>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared));
    k_radix_scatter<K><<<(unsigned)tiles, kSThreads, 0, st>>>(keys, out, count, shift, tiles, hist);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

// the passes from digit `shift` on, a -> b -> a ...
nd_status radix_passes(unsigned long long* a, unsigned long long* b, int64_t count, int shift, int bits, int64_t tiles,
                       int64_t* hist, unsigned long long** result, cudaStream_t st) {
    for (; shift < bits; shift += 8) {
        ND_TRY(radix_pass(KeyArray{a}, b, count, shift, tiles, hist, st));
        unsigned long long* t = a;
        a = b;
        b = t;
    }
    *result = a;
    return ND_OK;
}

}  // namespace

// stable LSD radix sort of keys[0, count) over their low `bits` bits; the
// result is in *result (keys or alt)
nd_status nd_sort_u64(unsigned long long* keys, unsigned long long* alt, int64_t count, int bits,
                      unsigned long long** result, cudaStream_t st) {
    *result = keys;
    if (count <= 1) return ND_OK;
    const int64_t tiles = (count + kTile - 1) / kTile;
    if (tiles > INT32_MAX) { nd_set_error("too many keys for one sort"); return ND_E_TOO_LARGE; }
    nd_tmp<int64_t> hist(st);
    ND_TRY(hist.alloc((int64_t)kBins * tiles + 1));
    return radix_passes(keys, alt, count, 0, bits, tiles, hist, result, st);
}

extern "C" nd_status nd_normalize(const int64_t* src, const int64_t* dst, int64_t m, int64_t n, int on_device,
                                  int64_t* row_ptr_out, int32_t* col_out, int64_t col_capacity, int64_t* nnz_out,
                                  void* stream) {
    if (m < 0 || n < 0 || col_capacity < 0) { nd_set_error("negative size"); return ND_E_INVAL; }
    if (n >= INT32_MAX) { nd_set_error("more than 2^31-1 vertices"); return ND_E_TOO_LARGE; }
    if (!nnz_out || !row_ptr_out || (m > 0 && (!src || !dst))) { nd_set_error("NULL argument"); return ND_E_INVAL; }
    if (m > 0 && n == 0) { nd_set_error("edges given for an empty vertex set"); return ND_E_INVAL; }
    *nnz_out = 0;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, sms = 152;
    ND_CUDA(cudaGetDevice(&dev));
    ND_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int bits = nd_id_bits(n);  // ids need `bits` bits; keys 2 * bits
    // device copies of host input
    const int64_t *dsrc = src, *ddst = dst;
    nd_tmp<int64_t> hsrc(st), hdst(st);
    if (!on_device && m > 0) {
        ND_TRY(hsrc.alloc(m));
        ND_TRY(hdst.alloc(m));
        ND_CUDA(cudaMemcpyAsync(hsrc, src, sizeof(int64_t) * m, cudaMemcpyHostToDevice, st));
        ND_CUDA(cudaMemcpyAsync(hdst, dst, sizeof(int64_t) * m, cudaMemcpyHostToDevice, st));
        dsrc = hsrc;
        ddst = hdst;
    }
    const int64_t count = 2 * m, tiles = (count + kTile - 1) / kTile;
    if (tiles > INT32_MAX) { nd_set_error("too many pairs for one sort"); return ND_E_TOO_LARGE; }
    nd_tmp<unsigned long long> keys(st), alt(st);
    nd_tmp<int64_t> hist(st), tile_first(st), before(st);
    nd_tmp<unsigned> first(st);
    nd_tmp<int> err(st);
    ND_TRY(keys.alloc(count));
    ND_TRY(alt.alloc(count));
    ND_TRY(hist.alloc((int64_t)kBins * tiles + 1));
    ND_TRY(tile_first.alloc(tiles + 1));
    ND_TRY(before.alloc((count + 31) / 32));
    ND_TRY(first.alloc((count + 31) / 32));
    ND_TRY(err.alloc(1));
    ND_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
    ND_CUDA(cudaMemsetAsync(tile_first.p + tiles, 0, sizeof(int64_t), st));
    unsigned long long* sorted = keys;
    if (m > 0) {
        ND_TRY(radix_pass(PairKeys{dsrc, ddst, n, bits, err}, keys.p, count, 0, tiles, hist, st));
        ND_TRY(radix_passes(keys, alt, count, 8, 2 * bits, tiles, hist, &sorted, st));
        nd_prof_scope ps("entry_bits", st);
        k_entry_bits<<<(unsigned)tiles, kThreads, 0, st>>>(sorted, count, bits, first, tile_first);
        ND_CUDA(cudaGetLastError());
    }
    ND_TRY(nd_scan_i64(tile_first, tiles, st));
    int64_t nnz = 0;
    int herr = 0;
    ND_CUDA(cudaMemcpyAsync(&nnz, tile_first.p + tiles, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    ND_CUDA(cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, st));
    ND_TRY(nd_wait(st));
    if (herr) { nd_set_error("a vertex id is outside [0, n)"); return ND_E_INVAL; }
    *nnz_out = nnz;
    if (nnz > col_capacity) {
        nd_set_error("col_out holds fewer entries than the normalised graph (*nnz_out gives the size needed)");
        return ND_E_INVAL;
    }
    if (nnz > 0 && !col_out) { nd_set_error("col_out is NULL"); return ND_E_INVAL; }
    // outputs: straight into device buffers, or staged for host buffers
    int32_t* dcol = col_out;
    int64_t* drp = row_ptr_out;
    nd_tmp<int32_t> scol(st);
    nd_tmp<int64_t> srp(st);
    if (!on_device) {
        ND_TRY(scol.alloc(nnz));
        ND_TRY(srp.alloc(n + 1));
        dcol = scol;
        drp = srp;
    }
    if (m > 0) {
        nd_prof_scope ps("write_entries", st);
        k_write_entries<<<(unsigned)tiles, kThreads, 0, st>>>(sorted, count, bits, first, tile_first, before, dcol);
        ND_CUDA(cudaGetLastError());
    }
    {
        nd_prof_scope ps("row_ptr", st);
        k_row_ptr<<<nd_blocks_for(n + 1, kThreads, sms * 8), kThreads, 0, st>>>(sorted, count, n, bits, first, before,
                                                                               nnz, drp);
        ND_CUDA(cudaGetLastError());
    }
    if (!on_device) {
        ND_CUDA(cudaMemcpyAsync(row_ptr_out, drp, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, st));
        if (nnz > 0) ND_CUDA(cudaMemcpyAsync(col_out, dcol, sizeof(int32_t) * nnz, cudaMemcpyDeviceToHost, st));
    }
    return nd_wait(st);
}
