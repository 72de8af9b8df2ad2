// Exclusive prefix sum of per-cell counts into cell offsets, over many CTAs
// (the grid builders' count -> start step). The number of cells lives on the
// device (the grid is set up there), so the host sizes the launches for an
// upper bound and CTAs past the real count return at once. Two launches:
//   scan_tile_sum_kernel: each CTA sums one tile of kScanTile counts;
//   scan_apply_kernel: each CTA adds up the sums of the tiles before its own,
//     scans its tile, writes the starts and zeroes the counts (the fill pass
//     counts again); the CTA of the last tile writes start[n] and calls the
//     finaliser with the total.
// Counts are int32, sums int64 (the bake checks the total against its entry
// capacity); starts are clamped to INT32_MAX.
#pragma once
#include <cstdint>

namespace sop {

constexpr int kScanThreads = 1024;
constexpr int kScanPer = 4;
constexpr int kScanTile = kScanThreads * kScanPer;

// tiles (CTAs) for at most n cells, and the int64 scratch the scan needs
inline unsigned scan_tiles(int64_t n) { return (unsigned)((n + kScanTile - 1) / kScanTile); }
inline size_t scan_scratch_count(int64_t n) { return (size_t)scan_tiles(n) + 2; }

struct ScanArgs {
    const int32_t* n;    // number of cells (device)
    int32_t* cnt;        // [n] counts (zeroed by the apply pass)
    int32_t* start;      // [n + 1] exclusive offsets
    long long* scratch;  // [tiles] sums
};

// inclusive block sum of one value per thread; returns it and leaves the
// block total in *total (shared scratch of kScanThreads / 32 entries)
static __device__ __forceinline__ long long scan_block_inclusive(long long v, long long* warp_sums, long long* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += u;
    }
    if (lane == 31) warp_sums[warp] = v;
    __syncthreads();
    if (warp == 0) {
        long long w = lane < kScanThreads / 32 ? warp_sums[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += u;
        }
        if (lane < kScanThreads / 32) warp_sums[lane] = w;
    }
    __syncthreads();
    const long long r = v + (warp > 0 ? warp_sums[warp - 1] : 0);
    *total = warp_sums[kScanThreads / 32 - 1];
    return r;
}

static __global__ void __launch_bounds__(kScanThreads) scan_tile_sum_kernel(ScanArgs a)
{
    __shared__ long long s_w[kScanThreads / 32];
    const int n = *a.n;
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    if (base >= n) return;
    long long v = 0;
#pragma unroll
    for (int e = 0; e < kScanPer; ++e) {
        const int64_t i = base + (int64_t)threadIdx.x * kScanPer + e;
        if (i < n) v += a.cnt[i];
    }
    long long tot;
    scan_block_inclusive(v, s_w, &tot);
    if (threadIdx.x == 0) a.scratch[blockIdx.x] = tot;
}

struct ScanNoFinal {
    __device__ void operator()(long long) const {}
};

template <class Fin>
static __global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(ScanArgs a, Fin fin)
{
    __shared__ long long s_w[kScanThreads / 32];
    const int n = *a.n;
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    if (base >= n) {
        if (n == 0 && blockIdx.x == 0 && threadIdx.x == 0) {  // no cells: start[0] = 0
            a.start[0] = 0;
            fin(0ll);
        }
        return;
    }
    int32_t c[kScanPer];
    long long v = 0;
#pragma unroll
    for (int e = 0; e < kScanPer; ++e) {
        const int64_t i = base + (int64_t)threadIdx.x * kScanPer + e;
        c[e] = i < n ? a.cnt[i] : 0;
        v += c[e];
    }
    long long before = 0, all, tot;
    for (int t = threadIdx.x; t < (int)blockIdx.x; t += kScanThreads) before += a.scratch[t];
    scan_block_inclusive(before, s_w, &all);
    __syncthreads();
    long long run = scan_block_inclusive(v, s_w, &tot) - v + all;
#pragma unroll
    for (int e = 0; e < kScanPer; ++e) {
        const int64_t i = base + (int64_t)threadIdx.x * kScanPer + e;
        if (i < n) {
            a.start[i] = (int32_t)(run < INT32_MAX ? run : INT32_MAX);
            a.cnt[i] = 0;
        }
        run += c[e];
    }
    if (base + kScanTile >= n && threadIdx.x == 0) {
        const long long total = all + tot;
        a.start[n] = (int32_t)(total < INT32_MAX ? total : INT32_MAX);
        fin(total);
    }
}

// the two launches for at most n_max cells
template <class Fin>
inline void launch_scan(const ScanArgs& a, int64_t n_max, Fin fin, cudaStream_t s)
{
    const unsigned nb = scan_tiles(n_max > 0 ? n_max : 1);
    scan_tile_sum_kernel<<<nb, kScanThreads, 0, s>>>(a);
    scan_apply_kernel<<<nb, kScanThreads, 0, s>>>(a, fin);
}

}  // namespace sop
