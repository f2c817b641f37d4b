// Exclusive prefix sums over int64 (offsets of every CSR this library builds).
//
// Two launches whatever the length: every block of a grid of at most
// kMaxBlocks sums its contiguous share of the array, then every block adds up
// the sums before its own (at most kMaxBlocks values, from L2) and scans its
// share tile by tile.  Arrays of a few tiles take the second launch alone.
// No recursion over tile sums, and no block waits for another.
// HBM-bound for long arrays: two reads and one write.  A recursive tile scan
// before: three launches, an allocation and a memset per level; a build of
// 10,000 edges spent 0.14 of its 1.1 ms in eight of them.
#include "nd_internal.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;
constexpr int kMaxBlocks = 608;   // 4 per SM of a 152-SM GPU; the second launch reads as many sums per block
constexpr int64_t kOneBlock = 4;  // tiles that one block scans alone

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// exclusive scan of one value per thread across the block, and the block's total
__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t& total) {
    __shared__ int64_t warp_sums[kThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t incl = warp_incl_scan(v);
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    int64_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        const int64_t s = warp_sums[w];
        if (w < wid) before += s;
        all += s;
    }
    __syncthreads();
    total = all;
    return before + incl - v;
}

// the kItems values of a thread from a[base]; base is a multiple of kItems
// and a comes from the allocator, so whole groups load as 16-byte pairs
__device__ __forceinline__ void load_items(const int64_t* __restrict__ a, int64_t base, int64_t n, int64_t (&v)[kItems]) {
    if (base + kItems <= n) {
        const longlong2* p = reinterpret_cast<const longlong2*>(a + base);
#pragma unroll
        for (int i = 0; i < kItems / 2; ++i) {
            const longlong2 x = p[i];
            v[2 * i] = x.x;
            v[2 * i + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kItems; ++i) v[i] = base + i < n ? a[base + i] : 0;
    }
}

// sums[b] = sum of block b's share, tiles [b * share, (b + 1) * share)
__global__ void __launch_bounds__(kThreads) k_share_sums(const int64_t* __restrict__ a, int64_t n, int64_t share,
                                                         int64_t* __restrict__ sums) {
    int64_t s = 0;
    for (int64_t t = 0; t < share; ++t) {
        const int64_t base = ((int64_t)blockIdx.x * share + t) * kTile + (int64_t)threadIdx.x * kItems;
        int64_t v[kItems];
        load_items(a, base, n, v);
#pragma unroll
        for (int i = 0; i < kItems; ++i) s += v[i];
    }
    int64_t total;
    block_excl_scan(s, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kThreads) k_share_scan(int64_t* __restrict__ a, int64_t n, int64_t share,
                                                         const int64_t* __restrict__ sums) {
    int64_t run = 0;
    if (sums) {
        int64_t s = 0, total;
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += kThreads) s += sums[i];
        block_excl_scan(s, total);
        run = total;
    }
    for (int64_t t = 0; t < share; ++t) {
        const int64_t tile = ((int64_t)blockIdx.x * share + t) * kTile;
        if (tile >= n) break;  // the same for the whole block
        const int64_t base = tile + (int64_t)threadIdx.x * kItems;
        int64_t v[kItems], s = 0, total;
        load_items(a, base, n, v);
#pragma unroll
        for (int i = 0; i < kItems; ++i) s += v[i];
        int64_t at = run + block_excl_scan(s, total);
        if (base + kItems <= n) {
            longlong2* p = reinterpret_cast<longlong2*>(a + base);
#pragma unroll
            for (int i = 0; i < kItems / 2; ++i) {
                p[i] = make_longlong2(at, at + v[2 * i]);
                at += v[2 * i] + v[2 * i + 1];
            }
        } else {
#pragma unroll
            for (int i = 0; i < kItems; ++i)
                if (base + i < n) {
                    a[base + i] = at;
                    at += v[i];
                }
        }
        run += total;
    }
}

}  // namespace

nd_status nd_scan_i64(int64_t* data, int64_t count, cudaStream_t st) {
    nd_prof_scope ps("scan", st);
    const int64_t n = count + 1;  // the trailing slot receives the total
    const int64_t tiles = (n + kTile - 1) / kTile;
    if (tiles <= kOneBlock) {
        k_share_scan<<<1, kThreads, 0, st>>>(data, n, tiles, nullptr);
        ND_CUDA(cudaGetLastError());
        return ND_OK;
    }
    const int64_t share = (tiles + kMaxBlocks - 1) / kMaxBlocks;
    const unsigned blocks = (unsigned)((tiles + share - 1) / share);
    nd_tmp<int64_t> sums(st);
    ND_TRY(sums.alloc(blocks));
    k_share_sums<<<blocks, kThreads, 0, st>>>(data, n, share, sums);
    ND_CUDA(cudaGetLastError());
    k_share_scan<<<blocks, kThreads, 0, st>>>(data, n, share, sums);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}
