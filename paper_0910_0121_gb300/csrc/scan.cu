// Device-wide exclusive prefix sum of uint32 arrays in one pass over them (tile_prefix),
// used for the node-ownership counts, the second-order lists and the domain counts.  The
// reduce-scan-scan form it replaced read the array twice in three launches or more: with
// the counters zeroed by earlier kernels and the group selection in one launch too, a call of
// 4 k particles took 0.182 ms where it had taken 0.225.
#include <algorithm>

#include "common.cuh"

namespace greem {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;  // 8 in single words: tree stage of 16.8 M particles 1.646 ms, 16 by 16-byte loads 1.535
constexpr int kScanTile = kScanThreads * kScanItems;

static inline size_t ceil_div(size_t a, size_t b) { return (a + b - 1) / b; }

// u32 words: the ticket, a pad, then one 64-bit look-back word per tile
size_t scan_zero_words(size_t n) { return 2 + 2 * std::max<size_t>(1, ceil_div(n, kScanTile)); }
size_t scan_scratch_elems(size_t n) { return scan_zero_words(n) + 2; }

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total)
{
    __shared__ uint32_t wsum[kScanThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t s = lane < kScanThreads / 32 ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kScanThreads / 32) wsum[lane] = s;
    }
    __syncthreads();
    uint32_t before = (w > 0 ? wsum[w - 1] : 0) + x - v;
    *total = wsum[kScanThreads / 32 - 1];
    __syncthreads();
    return before;
}

// Each thread owns kScanItems consecutive elements.
__global__ void __launch_bounds__(kScanThreads) k_scan(const uint32_t *in, size_t n, const uint32_t *__restrict__ n_dev,
                                                       uint32_t *out, uint32_t *scratch, DevStatus *st, uint32_t polls)
{
    __shared__ uint32_t s_tile, s_excl;
    if (threadIdx.x == 0) s_tile = atomicAdd(scratch, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (n_dev) n = min(n, (size_t)*n_dev);
    const size_t tbase = (size_t)tile * kScanTile;
    if (tbase >= n && tile > 0) return;
    const size_t base = tbase + (size_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
    const bool whole = base + kScanItems <= n;  // 16-byte loads and stores (in and out are 16-byte aligned)
    if (whole) {
#pragma unroll
        for (int t = 0; t < kScanItems; t += 4) {
            const uint4 u = *reinterpret_cast<const uint4 *>(in + base + t);
            v[t] = u.x;
            v[t + 1] = u.y;
            v[t + 2] = u.z;
            v[t + 3] = u.w;
        }
    } else {
#pragma unroll
        for (int t = 0; t < kScanItems; t++) v[t] = base + t < n ? in[base + t] : 0;
    }
#pragma unroll
    for (int t = 0; t < kScanItems; t++) s += v[t];
    uint32_t tot;
    uint32_t run = block_exclusive_scan(s, &tot);
    if (threadIdx.x < 32) {
        const uint32_t excl = tile_prefix(reinterpret_cast<unsigned long long *>(scratch + 2), tile, tot, st, polls);
        if (threadIdx.x == 0) s_excl = excl;
    }
    __syncthreads();
    run += s_excl;
#pragma unroll
    for (int t = 0; t < kScanItems; t++) {
        const uint32_t x = v[t];
        v[t] = run;
        run += x;
    }
    if (whole) {
#pragma unroll
        for (int t = 0; t < kScanItems; t += 4)
            *reinterpret_cast<uint4 *>(out + base + t) = make_uint4(v[t], v[t + 1], v[t + 2], v[t + 3]);
    } else {
#pragma unroll
        for (int t = 0; t < kScanItems; t++)
            if (base + t < n) out[base + t] = v[t];
    }
    // the thread holding element n-1 also writes the total at out[n]
    if (base < n && n - 1 < base + kScanItems) out[n] = run;
    if (n == 0 && threadIdx.x == 0) out[0] = 0;
}

void scan_u32(const uint32_t *in, uint32_t *out, size_t n, uint32_t *scratch, DevStatus *st, cudaStream_t s,
              const uint32_t *n_dev, bool zeroed, uint32_t polls)
{
    if (!zeroed) cudaMemsetAsync(scratch, 0, scan_zero_words(n) * sizeof(uint32_t), s);
    const unsigned nb = (unsigned)std::max<size_t>(1, ceil_div(n, kScanTile));
    k_scan<<<nb, kScanThreads, 0, s>>>(in, n, n_dev, out, scratch, st, polls);
    g_launches++;
}

}  // namespace greem
