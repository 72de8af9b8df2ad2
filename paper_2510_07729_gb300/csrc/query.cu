// SOP query + shade (Sec. 3.1.2 Eq. 2-6, Sec. 3.2.2 Eq. 7-9) for sm_103a.
//
// Launches of a query, in order:
//   query_tables_kernel  the probe grid (one CTA) beside the tables: light
//                        directions (Hammersley in fp64 -> fp32), bilinear
//                        footprints of the environment and of the atlas;
//   knn_warp_kernel /    exact K nearest probes by integer squared distance
//   knn_kernel           (rings of grid cells with an exact integer stopping
//                        bound), then the Eq. 4-6 weights; a warp or a
//                        thread a point;
//   one of               shade_kernel (LANES threads a point split the S
//                        directions, 4 texel fetches per probe and direction
//                        from the L2-resident footprints), shade_point_kernel
//                        (a warp a point, probes blended first),
//                        shadow_warp_kernel (SHADOW: points on one normal
//                        share each probe's integral), shade_world_kernel
//                        (importance-sampled directions).
#include <float.h>
#include <stdlib.h>

#include <mutex>

#include "point_blend.cuh"
#include "scan.cuh"
#include "sop_device.cuh"
#include "sop_internal.h"

namespace sop {

QueryLayout query_layout(int32_t P, int64_t M, int32_t K, int32_t S, int32_t He, int32_t We, int32_t R,
                         int32_t rgbo_dtype)
{
    QueryLayout L{};
    int g = 1;
    while ((int64_t)g * g * g < P) ++g;
    L.g_axis = g;
    L.cells_cap = (g + 1) * (g + 1) * (g + 1);
    size_t o = 0;
    L.grid_hdr = o;   o = align256(o + sizeof(ProbeGrid));
    L.cell_start = o; o = align256(o + sizeof(int32_t) * (size_t)(L.cells_cap + 1));
    L.cell_cnt = o;   o = align256(o + sizeof(int32_t) * (size_t)L.cells_cap);
    L.entries = o;    o = align256(o + sizeof(int4) * (size_t)P);
    L.envq = o;       o = align256(o + 64 * (size_t)(He + 1) * (We + 1));  // both layouts
    L.quads = o;      o = align256(o + (rgbo_dtype == SOP_F32 ? 64 : 32) * (size_t)P * (R + 1) * (R + 1));
    L.dirs = o;       o = align256(o + sizeof(float4) * (size_t)S);
    L.idx = o;        o = align256(o + sizeof(int32_t) * (size_t)M * K);
    L.w = o;          o = align256(o + sizeof(float) * (size_t)M * K);
    // adjoint only: points grouped by nearest probe, and the environment
    // gradient as float4 texels
    L.perm = o;       o = align256(o + sizeof(int32_t) * (size_t)M);
    L.bucket = o;     o = align256(o + sizeof(int32_t) * (size_t)(P + 1));
    L.genv4 = o;      o = align256(o + sizeof(float4) * (size_t)He * We);
    L.total = o;
    return L;
}

__device__ __forceinline__ int32_t quantise(float v) { return __float2int_rn(v * 1048576.0f); }

// Exact squared distance of two quantised points. Coordinates are below 2^30
// in magnitude (positions below 1024), so each difference fits 32 bits and
// each square is one 32x32 -> 64-bit multiply; the sum stays below 3 * 2^62.
__device__ __forceinline__ uint64_t qdist2(int32_t ax, int32_t ay, int32_t az, const int32_t q[3])
{
    const uint32_t dx = (uint32_t)abs(ax - q[0]), dy = (uint32_t)abs(ay - q[1]), dz = (uint32_t)abs(az - q[2]);
    return (uint64_t)dx * dx + (uint64_t)dy * dy + (uint64_t)dz * dz;
}

// cell of a site of the set (quantised position), by the grid's edge
__device__ __forceinline__ int grid_cell(const ProbeGrid& G, int32_t qx, int32_t qy, int32_t qz)
{
    const uint32_t cs = (uint32_t)G.cs;
    const int cx = (int)div_by((uint32_t)qx - (uint32_t)G.qmin[0], cs, G.inv);
    const int cy = (int)div_by((uint32_t)qy - (uint32_t)G.qmin[1], cs, G.inv);
    const int cz = (int)div_by((uint32_t)qz - (uint32_t)G.qmin[2], cs, G.inv);
    return (cz * G.dims[1] + cy) * G.dims[0] + cx;
}

// ---------------------------------------------------------------------------
// Probe grid, built by one CTA of 1,024 threads (P is small: thousands to
// ~1e5 probes). A serial chain of short steps, so each is kept short: the
// candidate edges of all five coarsening levels are searched at once, a warp
// each, 32 edges a step; cells are counted, scanned and filled in shared
// memory while they fit (kGridSmemCells); divisions by the edge are one
// multiplication. 4,096 probes: 26-49 us when one thread bisected each edge
// by 64-bit divisions and the cells were counted in memory; with all of a
// query's tables beside it 16-20 us now.
// ---------------------------------------------------------------------------
constexpr int kGridThreads = 1024;
constexpr int kGridLevels = 5;
constexpr int kGridSmemCells = 8192;

struct GridSmem {
    int32_t mn[3], mx[3];
    uint32_t edge[kGridLevels];
    int32_t occ;
    int32_t warp[32];
    int32_t cnt[kGridSmemCells];
};

// Cells of edge e over a box of extents ext; at most cap?
__device__ __forceinline__ bool grid_fits(const uint32_t ext[3], uint64_t e, int64_t cap)
{
    uint64_t n = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        n *= (e > ext[a] ? 0u : ext[a] / (uint32_t)e) + 1u;
        if (n > (uint64_t)cap) return false;
    }
    return true;
}

// Smallest edge (quantised units) that fits, by one warp, 32 candidates a step.
// A flat site set (probes on a ground plane) then gets fine cells in its
// plane instead of the cbrt-per-axis split of a volume, which would put
// cbrt(P) sites in every cell of its one layer.
__device__ __forceinline__ uint32_t grid_edge(const uint32_t ext[3], const int64_t cap, const int lane)
{
    uint64_t lo = 1, hi = (uint64_t)max(ext[0], max(ext[1], ext[2])) + 1;  // hi: one cell per axis
    while (lo < hi) {
        const uint64_t step = (hi - lo + 31) / 32, e = min(lo + lane * step, hi);
        const unsigned ok = __ballot_sync(0xffffffffu, grid_fits(ext, e, cap));
        const int f = ok ? __ffs(ok) - 1 : 32;
        if (f == 0) hi = lo;
        else {
            if (f < 32) hi = min(lo + f * step, hi);
            lo = min(lo + (f - 1) * step, hi) + 1;
        }
    }
    // (an edge of 2^31 and more: one cell per axis too)
    return (uint32_t)min(lo, (uint64_t)INT32_MAX);
}

__device__ __forceinline__ void probe_grid_build(GridSmem& sm, const float* __restrict__ probe_pos, int32_t P,
                                                 int32_t g_axis, ProbeGrid* grid, int32_t* cell_start,
                                                 int32_t* cell_cnt, int4* entries)
{
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, nt = kGridThreads, lane = tid & 31, warp = tid >> 5;
    if (tid < 3) {
        sm.mn[tid] = INT32_MAX;
        sm.mx[tid] = INT32_MIN;
    }
    __syncthreads();
    int32_t lmin[3] = {INT32_MAX, INT32_MAX, INT32_MAX}, lmax[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
    for (int p = tid; p < P; p += nt)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int32_t q = quantise(probe_pos[3 * p + a]);
            lmin[a] = min(lmin[a], q);
            lmax[a] = max(lmax[a], q);
        }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int32_t lo = __reduce_min_sync(full, lmin[a]), hi = __reduce_max_sync(full, lmax[a]);
        if (lane == 0 && lo <= hi) {
            atomicMin(&sm.mn[a], lo);
            atomicMax(&sm.mx[a], hi);
        }
    }
    __syncthreads();
    // cell edge: the finest grid within (g+1)^3 cells, coarsened (cap
    // halved, at most 4 times) while there are fewer than 3 probes per
    // occupied cell. A volume-like set keeps the fine grid; a flat one (the
    // shadow probes on the ground), whose far query points need the K
    // nearest from a wide strip, gets cells of a few probes each.
    const int64_t cap0 = (int64_t)(g_axis + 1) * (g_axis + 1) * (g_axis + 1);
    uint32_t ext[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) ext[a] = (uint32_t)sm.mx[a] - (uint32_t)sm.mn[a];
    if (warp < kGridLevels) {
        const uint32_t e = grid_edge(ext, cap0 >> warp, lane);
        if (lane == 0) sm.edge[warp] = e;
    }
    __syncthreads();
    const bool in_smem = cap0 <= kGridSmemCells;
    int32_t* cnt = in_smem ? sm.cnt : cell_cnt;
    ProbeGrid G;
    for (int it = 0;; ++it) {
        const uint32_t cs = sm.edge[it];
        G.cs = (int32_t)cs;
        G.inv = 0xffffffffu / cs;
        G.ncells = 1;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            G.qmin[a] = sm.mn[a];
            G.dims[a] = (int32_t)(ext[a] / cs) + 1;
            G.ncells *= G.dims[a];
        }
        if (tid == 0) sm.occ = 0;
        for (int c = tid; c < G.ncells; c += nt) cnt[c] = 0;
        __syncthreads();
        int occ = 0;
        for (int p = tid; p < P; p += nt)
            if (atomicAdd(&cnt[grid_cell(G, quantise(probe_pos[3 * p]), quantise(probe_pos[3 * p + 1]),
                                         quantise(probe_pos[3 * p + 2]))], 1) == 0)
                ++occ;
        occ = __reduce_add_sync(full, occ);
        if (lane == 0 && occ) atomicAdd(&sm.occ, occ);
        __syncthreads();
        const bool again = it < kGridLevels - 1 && (int64_t)P < 3 * (int64_t)sm.occ && (cap0 >> it) > 8;
        __syncthreads();
        if (!again) break;
    }
    if (tid == 0) *grid = G;
    // exclusive scan of the counts: a contiguous chunk per thread, then the block
    const int nc = G.ncells, chunk = (nc + nt - 1) / nt;
    const int c0 = min(nc, tid * chunk), c1 = min(nc, c0 + chunk);
    int32_t sum = 0;
    for (int c = c0; c < c1; ++c) sum += cnt[c];
    int32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t v = __shfl_up_sync(full, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) sm.warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int32_t w = sm.warp[lane];
        int32_t v = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(full, v, o);
            if (lane >= o) v += u;
        }
        sm.warp[lane] = v - w;
    }
    __syncthreads();
    int32_t run = inc - sum + sm.warp[warp];
    for (int c = c0; c < c1; ++c) {
        const int32_t v = cnt[c];
        cell_start[c] = run;
        cnt[c] = in_smem ? run : 0;  // the fill's cursor
        run += v;
    }
    if (tid == nt - 1) cell_start[nc] = P;
    __syncthreads();
    for (int p = tid; p < P; p += nt) {
        const int32_t qx = quantise(probe_pos[3 * p]), qy = quantise(probe_pos[3 * p + 1]),
                      qz = quantise(probe_pos[3 * p + 2]);
        const int cell = grid_cell(G, qx, qy, qz);
        const int at = atomicAdd(&cnt[cell], 1) + (in_smem ? 0 : cell_start[cell]);
        entries[at] = make_int4(qx, qy, qz, p);
    }
}

__global__ void __launch_bounds__(kGridThreads) probe_grid_kernel(const float* __restrict__ probe_pos, int32_t P,
                                                                  int32_t g_axis, ProbeGrid* grid, int32_t* cell_start,
                                                                  int32_t* cell_cnt, int4* entries)
{
    __shared__ GridSmem sm;
    probe_grid_build(sm, probe_pos, P, g_axis, grid, cell_start, cell_cnt, entries);
}

// the point's cell along one axis, clamped into the grid
__device__ __forceinline__ int grid_axis_cell(const ProbeGrid& G, int a, int32_t q)
{
    if (q < G.qmin[a]) return 0;
    return min((int)div_by((uint32_t)q - (uint32_t)G.qmin[a], (uint32_t)G.cs, G.inv), G.dims[a] - 1);
}

// The search visits rings of cells (Chebyshev radius r in cell indices)
// around cc, the point's cell clamped into the grid. This is a lower bound on
// the squared quantised distance from the point q to every cell outside the
// cube of radius r: an unsearched cell lies in a slab beyond the cube along
// some axis b (below cc_b - r or above cc_b + r), at least d_b away along b,
// and, being inside the grid, at least out_a away along every other axis a
// (out_a: the point's distance outside the grid's extent on axis a; 0 for a
// point within it). The bound is the smallest d_b^2 + sum_{a != b} out_a^2
// over the slabs that hold cells; UINT64_MAX once the cube covers the grid.
// A site whose key is below it has been seen; sums that overflow 64 bits
// exceed every key and saturate.
__device__ __forceinline__ uint64_t unsearched_bound2(const ProbeGrid& G, const int32_t q[3], const int cc[3], int r)
{
    uint64_t out2[3], osum = 0;
    for (int a = 0; a < 3; ++a) {
        const int64_t lo = G.qmin[a], hi = lo + (int64_t)G.dims[a] * G.cs;
        const int64_t o = q[a] < lo ? lo - q[a] : (q[a] >= hi ? q[a] - hi + 1 : 0);
        out2[a] = (uint64_t)(o * o);
        osum += out2[a];
    }
    uint64_t best = UINT64_MAX;
    for (int b = 0; b < 3; ++b) {
        const uint64_t rest = osum - out2[b];
        // d^2 + rest, unless it exceeds 64 bits (then it bounds nothing)
        auto take = [&](uint64_t d) {
            if (d >> 32) return;
            const uint64_t v = (uint64_t)(uint32_t)d * (uint32_t)d + rest;
            if (v >= rest && v < best) best = v;
        };
        // cells of index <= cc_b - r - 1 end at qmin + (cc_b - r) cs
        if (cc[b] - r > 0) take((uint64_t)((int64_t)q[b] - (G.qmin[b] + (int64_t)(cc[b] - r) * G.cs)));
        // cells of index >= cc_b + r + 1 start at qmin + (cc_b + r + 1) cs
        if (cc[b] + r < G.dims[b] - 1) take((uint64_t)((G.qmin[b] + (int64_t)(cc[b] + r + 1) * G.cs) - (int64_t)q[b]));
    }
    return best;
}

// ---------------------------------------------------------------------------
// Exact K nearest probes + blend weights. One thread per point.
// Bound: the ALU pipe (64-bit keys). A (key, index) pair fits one 64-bit word
// where the point's largest possible key leaves room for the index (PACKED:
// 4,096 probes within 64 units): comparing and moving a kept pair is then 6
// instructions instead of 10. A cell whose nearest point lies beyond the K-th
// kept key is not read. 2,051,693 pixels of a ground frame, 4,096 probes,
// K = 8: 497 -> 405 us (5,290 instructions a warp); an object view of 418,111:
// 178 -> 155 us. K 5 to 8: nine CTAs an SM (56 registers, 24 bytes spilled)
// instead of eight: the frame's whole call 694 -> 678 us, ten (48, 88 bytes):
// 680. Up to K 4 eight (64 registers): searches of 2,051,693 ground points 383
// us with nine, 368 with eight, 377 with ten, 391 unbounded (K 1: 276 / 264 /
// 273 / 282; 418,111 points of an object 158 / 155 / 160 / 161).
// ---------------------------------------------------------------------------
// squared distance along one axis from q to the cell interval [lo, lo + cs)
__device__ __forceinline__ uint64_t axis_gap2(int32_t q, int64_t lo, int32_t cs)
{
    const int64_t a = lo - q, b = (int64_t)q - (lo + cs - 1), g = a > 0 ? a : (b > 0 ? b : 0);
    if (g >> 32) return UINT64_MAX;  // (never for positions below 1024)
    return (uint64_t)(uint32_t)g * (uint32_t)g;
}

// The KMAX best pairs, sorted, into bk and bi (bi = INT32_MAX where fewer lie
// within the radius); the first K of them are exact.
template <int KMAX, bool PACKED>
__device__ __forceinline__ void knn_search(const ProbeGrid& G, const int32_t q[3], int K, uint64_t r2_key, int id_bits,
                                           const int32_t* __restrict__ cell_start, const int4* __restrict__ entries,
                                           uint64_t* bk, int32_t* bi)
{
    // rings are taken around the point's cell clamped into the grid
    const int c[3] = {grid_axis_cell(G, 0, q[0]), grid_axis_cell(G, 1, q[1]), grid_axis_cell(G, 2, q[2])};
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        bk[k] = UINT64_MAX;
        if (!PACKED) bi[k] = INT32_MAX;
    }
    // the K-th best key as a chain of selects: picking bk[K - 1] by the
    // run-time K would put bk in local memory
    const auto kth_key = [&]() {
        uint64_t v = bk[0];
#pragma unroll
        for (int k = 1; k < KMAX; ++k) v = k < K ? bk[k] : v;
        return PACKED && v != UINT64_MAX ? v >> id_bits : v;
    };
    for (int r = 0;; ++r) {
        const uint64_t kth0 = kth_key(), lim = kth0 < r2_key ? kth0 : r2_key;
        const int zlo = max(c[2] - r, 0), zhi = min(c[2] + r, G.dims[2] - 1);
        const int ylo = max(c[1] - r, 0), yhi = min(c[1] + r, G.dims[1] - 1);
        for (int z = zlo; z <= zhi; ++z) {
            const uint64_t gz = axis_gap2(q[2], G.qmin[2] + (int64_t)z * G.cs, G.cs);
            if (gz > lim) continue;
            for (int y = ylo; y <= yhi; ++y) {
                const uint64_t gyz = gz + axis_gap2(q[1], G.qmin[1] + (int64_t)y * G.cs, G.cs);
                if (gyz > lim) continue;
                const bool face = (z == c[2] - r) || (z == c[2] + r) || (y == c[1] - r) || (y == c[1] + r);
                const int xs = face ? 1 : 2 * r;  // on a face row: every x; else only the two ends
                for (int xx = c[0] - r; xx <= c[0] + r; xx += (xs > 0 ? xs : 1)) {
                    if (xx < 0 || xx >= G.dims[0]) continue;
                    if (gyz + axis_gap2(q[0], G.qmin[0] + (int64_t)xx * G.cs, G.cs) > lim) continue;
                    const int cell = (z * G.dims[1] + y) * G.dims[0] + xx;
                    const int e1 = __ldg(cell_start + cell + 1);
#pragma unroll 2
                    for (int e = __ldg(cell_start + cell); e < e1; ++e) {
                        const int4 en = __ldg(entries + e);
                        const uint64_t key = qdist2(en.x, en.y, en.z, q);
                        // keep the KMAX best pairs within the radius sorted;
                        // the first K of them are the K nearest. Insert: every
                        // kept pair above the new one moves up a slot
                        bool lt[KMAX];
                        if (PACKED) {
                            const uint64_t kp = key << id_bits | (uint32_t)en.w;
                            if (!(key <= r2_key && kp < bk[KMAX - 1])) continue;
#pragma unroll
                            for (int k = 0; k < KMAX; ++k) lt[k] = kp < bk[k];
#pragma unroll
                            for (int k = KMAX - 1; k > 0; --k) bk[k] = lt[k - 1] ? bk[k - 1] : (lt[k] ? kp : bk[k]);
                            bk[0] = lt[0] ? kp : bk[0];
                        } else {
                            const int32_t id = en.w;
                            if (!(key <= r2_key && (key < bk[KMAX - 1] || (key == bk[KMAX - 1] && id < bi[KMAX - 1]))))
                                continue;
#pragma unroll
                            for (int k = 0; k < KMAX; ++k) lt[k] = key < bk[k] || (key == bk[k] && id < bi[k]);
#pragma unroll
                            for (int k = KMAX - 1; k > 0; --k) {
                                bk[k] = lt[k - 1] ? bk[k - 1] : (lt[k] ? key : bk[k]);
                                bi[k] = lt[k - 1] ? bi[k - 1] : (lt[k] ? id : bi[k]);
                            }
                            bk[0] = lt[0] ? key : bk[0];
                            bi[0] = lt[0] ? id : bi[0];
                        }
                    }
                }
            }
        }
        // stop once no probe outside ring r can enter the best K, nor lie
        // within the radius
        const uint64_t bnd = unsearched_bound2(G, q, c, r);
        if (bnd == UINT64_MAX || kth_key() < bnd || r2_key < bnd) break;
    }
    if (PACKED)
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            const bool on = bk[k] != UINT64_MAX;
            bi[k] = on ? (int32_t)(bk[k] & ((1ull << id_bits) - 1ull)) : INT32_MAX;
            bk[k] = on ? bk[k] >> id_bits : UINT64_MAX;
        }
}

template <int KMAX>
__global__ void __launch_bounds__(128, KMAX <= 4 ? 8 : (KMAX <= 8 ? 9 : 1)) knn_kernel(const float* __restrict__ x, const float* __restrict__ nrm, int64_t M,
                                                   int32_t K, int32_t id_bits, uint64_t snap_key, uint64_t r2_key,
                                                   const ProbeGrid* __restrict__ gridp,
                                                   const int32_t* __restrict__ cell_start,
                                                   const int4* __restrict__ entries,
                                                   const float* __restrict__ probe_pos, int32_t* __restrict__ ws_idx,
                                                   float* __restrict__ ws_w, int32_t* __restrict__ user_idx,
                                                   float* __restrict__ user_w, unsigned int* status)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const ProbeGrid G = *gridp;
    float3 xp = load3(x, m);
    {
        // a non-finite position or normal is reported; the position is then
        // taken as the origin so that the search stays defined
        const float3 nr0 = load3(nrm, m);
        const bool okx = isfinite(xp.x + xp.y + xp.z);
        if ((!okx || !isfinite(nr0.x + nr0.y + nr0.z)) && status) atomicOr(status, SOP_DEVSTAT_NONFINITE);
        if (!okx) xp = f3(0.f, 0.f, 0.f);
    }
    const int32_t q[3] = {quantise(xp.x), quantise(xp.y), quantise(xp.z)};
    uint64_t bk[KMAX];
    int32_t bi[KMAX];
    // the largest key a probe of the grid's box can have (each term below
    // 2^62 when its distance is below 2^31)
    uint64_t far2 = 0;
    bool room = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int64_t lo = G.qmin[a], hi = lo + (int64_t)G.dims[a] * G.cs;
        const int64_t d = max(llabs(q[a] - lo), llabs(q[a] - hi));
        room = room && d < ((int64_t)1 << 30);
        far2 += (uint64_t)d * (uint64_t)d;
    }
    // (all ones is the empty slot, so the largest pair stays below it)
    room = room && (far2 >> (63 - id_bits)) == 0;
    if (__all_sync(__activemask(), room))
        knn_search<KMAX, true>(G, q, K, r2_key, id_bits, cell_start, entries, bk, bi);
    else knn_search<KMAX, false>(G, q, K, r2_key, id_bits, cell_start, entries, bk, bi);
    // weights (Eq. 4-6)
    const float3 nr = load3(nrm, m);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 nn = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    float w[KMAX];
    float wsum = 0.f;
    // slots a radius search left empty keep bi = INT32_MAX: weight 0, and the
    // shading reads (with weight 0) the nearest probe found, or probe 0
    const bool snap = bi[0] != INT32_MAX && bk[0] <= snap_key;
    const int32_t fill = bi[0] != INT32_MAX ? bi[0] : 0;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        w[k] = 0.f;
        if (k < K && bi[k] != INT32_MAX) {
            const float3 pk = load3(probe_pos, bi[k]);
            const float3 d = pk - xp;
            const float dl = sqrtf(dot3(d, d));
            const float ws = 1.f / dl;
            const float wb = 0.5f * (1.f + dot3(d, nn) / dl) + 0.01f;
            w[k] = snap ? (k == 0 ? 1.f : 0.f) : ws * wb;
            wsum += w[k];
        }
    }
#pragma unroll
    for (int k = 0; k < KMAX; ++k)
        if (k < K) {
            const bool found = bi[k] != INT32_MAX;
            const float wk = (snap || !found) ? w[k] : w[k] / wsum;
            ws_idx[m * K + k] = found ? bi[k] : fill;
            ws_w[m * K + k] = wk;
            if (user_idx) user_idx[m * K + k] = found ? bi[k] : -1;
            if (user_w) user_w[m * K + k] = wk;
        }
}

// ---------------------------------------------------------------------------
// The same search, one warp per point, for calls that do not fill the machine
// with a thread a point: a thread's search is a chain of dependent loads
// (cell, entries, insertion) of 20 to 60 us however few points there are. The
// lanes take the cells of the cube around the point, 32 at a time, and their
// entries side by side; candidates gather in shared memory and the K best are
// picked by warp minima. With few probes (entries NULL) the lanes take all of
// them and no grid is needed.
// ---------------------------------------------------------------------------
constexpr int kKnnWarps = 8;
constexpr int kKnnBuf = 128;  // candidates a warp holds

struct KnnK {
    const float *x, *nrm;
    int64_t M;
    int32_t K, P;
    uint64_t snap_key, r2_key;
    const ProbeGrid* grid;
    const int32_t* cell_start;
    const int4* entries;
    const float* probe_pos;
    int32_t* ws_idx;
    float* ws_w;
    int32_t* user_idx;
    float* user_w;
    unsigned int* status;
};

// The K best of the cnt candidates, sorted, to the front; returns their number.
__device__ __forceinline__ int knn_select(uint64_t* key, int32_t* id, int cnt, int K, int lane)
{
    constexpr int PER = kKnnBuf / 32;
    const unsigned full = 0xffffffffu;
    uint64_t lk[PER];
    int32_t li[PER];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const bool on = j * 32 + lane < cnt;
        lk[j] = on ? key[j * 32 + lane] : UINT64_MAX;
        li[j] = on ? id[j * 32 + lane] : INT32_MAX;
    }
    __syncwarp();
    const int n = min(K, cnt);
    for (int r = 0; r < n; ++r) {
        uint64_t bk = lk[0];
        int32_t bi = li[0];
#pragma unroll
        for (int j = 1; j < PER; ++j) {
            const bool lt = lk[j] < bk || (lk[j] == bk && li[j] < bi);
            bk = lt ? lk[j] : bk;
            bi = lt ? li[j] : bi;
        }
        const uint32_t hi = __reduce_min_sync(full, (uint32_t)(bk >> 32));
        const uint32_t lo = __reduce_min_sync(full, (uint32_t)(bk >> 32) == hi ? (uint32_t)bk : 0xffffffffu);
        const uint64_t wk = (uint64_t)hi << 32 | lo;
        const int32_t wi = (int32_t)__reduce_min_sync(full, bk == wk ? (uint32_t)bi : (uint32_t)INT32_MAX);
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (lk[j] == wk && li[j] == wi) {
                lk[j] = UINT64_MAX;
                li[j] = INT32_MAX;
            }
        if (lane == 0) {
            key[r] = wk;
            id[r] = wi;
        }
    }
    __syncwarp();
    return n;
}

__global__ void __launch_bounds__(kKnnWarps * 32) knn_warp_kernel(const KnnK a)
{
    __shared__ uint64_t s_key[kKnnWarps][kKnnBuf];
    __shared__ int32_t s_id[kKnnWarps][kKnnBuf];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t m = (int64_t)blockIdx.x * kKnnWarps + warp;
    if (m >= a.M) return;
    uint64_t* key = s_key[warp];
    int32_t* id = s_id[warp];
    const int K = a.K;
    float3 xp = load3(a.x, m);
    const float3 nr = load3(a.nrm, m);
    const bool okx = isfinite(xp.x + xp.y + xp.z);
    if (lane == 0 && (!okx || !isfinite(nr.x + nr.y + nr.z)) && a.status) atomicOr(a.status, SOP_DEVSTAT_NONFINITE);
    if (!okx) xp = f3(0.f, 0.f, 0.f);
    const int32_t q[3] = {quantise(xp.x), quantise(xp.y), quantise(xp.z)};
    int cnt = 0;
    uint64_t kth = UINT64_MAX;  // no candidate above it can be among the K
    const auto add = [&](bool on, int4 en) {
        const uint64_t k = on ? qdist2(en.x, en.y, en.z, q) : UINT64_MAX;
        const bool pass = on && k <= a.r2_key && k <= kth;
        const unsigned pm = __ballot_sync(full, pass);
        if (pass) {
            const int at = cnt + __popc(pm & ((1u << lane) - 1u));
            key[at] = k;
            id[at] = en.w;
        }
        cnt += __popc(pm);
        if (cnt > kKnnBuf - 32) {
            cnt = knn_select(key, id, cnt, K, lane);
            kth = cnt == K ? key[K - 1] : UINT64_MAX;
        }
    };
    if (!a.entries) {
        for (int p0 = 0; p0 < a.P; p0 += 32) {
            const int p = min(p0 + lane, a.P - 1);
            add(p0 + lane < a.P, make_int4(quantise(__ldg(a.probe_pos + 3 * p)), quantise(__ldg(a.probe_pos + 3 * p + 1)),
                                           quantise(__ldg(a.probe_pos + 3 * p + 2)), p));
        }
        cnt = knn_select(key, id, cnt, K, lane);
    } else {
        const ProbeGrid G = *a.grid;
        const int c[3] = {grid_axis_cell(G, 0, q[0]), grid_axis_cell(G, 1, q[1]), grid_axis_cell(G, 2, q[2])};
        // cubes of radius 1, 2, ... cells (each without the one before)
        for (int r = 1;; ++r) {
            const int x0 = max(c[0] - r, 0), y0 = max(c[1] - r, 0), z0 = max(c[2] - r, 0);
            const int nx = min(c[0] + r, G.dims[0] - 1) - x0 + 1, ny = min(c[1] + r, G.dims[1] - 1) - y0 + 1,
                      nz = min(c[2] + r, G.dims[2] - 1) - z0 + 1, nc = nx * ny * nz;
            for (int l0 = 0; l0 < nc; l0 += 32) {
                const int l = l0 + lane;
                const int xx = x0 + l % nx, yz = l / nx, yy = y0 + yz % ny, zz = z0 + yz / ny;
                const int far = max(max(abs(xx - c[0]), abs(yy - c[1])), abs(zz - c[2]));
                int e = 0, e1 = 0;
                if (l < nc && (r == 1 || far == r)) {
                    const int cell = (zz * G.dims[1] + yy) * G.dims[0] + xx;
                    e = __ldg(a.cell_start + cell);
                    e1 = __ldg(a.cell_start + cell + 1);
                }
                while (__any_sync(full, e < e1)) {
                    const bool on = e < e1;
                    add(on, on ? __ldg(a.entries + e) : make_int4(0, 0, 0, 0));
                    ++e;
                }
            }
            cnt = knn_select(key, id, cnt, K, lane);
            kth = cnt == K ? key[K - 1] : UINT64_MAX;
            const uint64_t bnd = unsearched_bound2(G, q, c, r);
            if (bnd == UINT64_MAX || kth < bnd || a.r2_key < bnd) break;
        }
    }
    // weights (Eq. 4-6), lane k for neighbour k; the same arithmetic and order
    // of the sum as knn_kernel
    const float nl = sqrtf(dot3(nr, nr));
    const float3 nn = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    const bool found = lane < cnt;
    const int32_t bi = found ? id[lane] : 0;
    const bool snap = cnt > 0 && key[0] <= a.snap_key;
    const int32_t fill = cnt > 0 ? id[0] : 0;
    float w = 0.f;
    if (found) {
        const float3 d = load3(a.probe_pos, bi) - xp;
        const float dl = sqrtf(dot3(d, d));
        const float ws = 1.f / dl;
        const float wb = 0.5f * (1.f + dot3(d, nn) / dl) + 0.01f;
        w = snap ? (lane == 0 ? 1.f : 0.f) : ws * wb;
    }
    float wsum = 0.f;
    for (int k = 0; k < cnt; ++k) wsum += __shfl_sync(full, w, k);
    if (lane < K) {
        const float wk = (snap || !found) ? w : w / wsum;
        a.ws_idx[m * K + lane] = found ? bi : fill;
        a.ws_w[m * K + lane] = wk;
        if (a.user_idx) a.user_idx[m * K + lane] = found ? bi : -1;
        if (a.user_w) a.user_w[m * K + lane] = wk;
    }
}

// ---------------------------------------------------------------------------
// Tables of a query, all in one launch with the probe grid (query_tables_kernel):
// the environment's and the atlas's bilinear footprints, and the directions.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void flag_nonfinite(bool ok, unsigned int* status)
{
    if (!ok && status) atomicOr(status, SOP_DEVSTAT_NONFINITE);
}

// Environment footprints: for base (r0, c0), r0 in [0, He], c0 in [0, We),
// the 2x2 bilinear footprint of rows r0 - 1, r0 (clamped) and columns c0,
// c0 + 1 (wrapped), RGB x 4 = 12 floats in a 64-byte slot: (e00, e01, e10,
// e11) with e01 the next column, e10 the next row.
__device__ __forceinline__ void env_footprint(const float* __restrict__ env, int32_t He, int32_t We, int64_t i,
                                              float4* __restrict__ envq, unsigned int* status)
{
    const int r0 = (int)(i / We), c0 = (int)(i % We), c1 = c0 + 1 == We ? 0 : c0 + 1;
    const int ra = max(r0 - 1, 0), rb = min(r0, He - 1);
    const float3 a = load3(env, (int64_t)ra * We + c0), b = load3(env, (int64_t)ra * We + c1),
                 c = load3(env, (int64_t)rb * We + c0), d = load3(env, (int64_t)rb * We + c1);
    flag_nonfinite(isfinite(c.x + c.y + c.z), status);  // (r0 < He covers every texel)
    float4* q = envq + 4 * i;
    q[0] = make_float4(a.x, a.y, a.z, b.x);
    q[1] = make_float4(b.y, b.z, c.x, c.y);
    q[2] = make_float4(c.z, d.x, d.y, d.z);
    q[3] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Octahedral environment footprints (Sec. 4.1 layout, [H][H][3]): for base
// (a, b) in [0, H]^2, the texels (a-1+di, b-1+dj), di, dj in {0, 1}, through
// the probe maps' border rule, in the same slots.
__device__ __forceinline__ void env_oct_footprint(const float* __restrict__ env, int32_t H, int64_t k,
                                                  float4* __restrict__ envq, unsigned int* status)
{
    const int HQ = H + 1;
    const int b = (int)(k / HQ), a = (int)(k % HQ);
    float3 e[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int si, sj;
        oct_wrap(H, a - 1 + (q & 1), b - 1 + (q >> 1), si, sj);
        e[q] = load3(env, (int64_t)sj * H + si);
    }
    flag_nonfinite(isfinite(e[0].x + e[0].y + e[0].z), status);
    float4* o = envq + 4 * k;
    o[0] = make_float4(e[0].x, e[0].y, e[0].z, e[1].x);
    o[1] = make_float4(e[1].y, e[1].z, e[2].x, e[2].y);
    o[2] = make_float4(e[2].z, e[3].x, e[3].y, e[3].z);
    o[3] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Atlas footprints: for probe p and base (a, b) in [0, R]^2 of the stored
// (gutter) map, the texels (a,b), (a+1,b), (a,b+1), (a+1,b+1) stored
// contiguously, so one bilinear fetch reads one aligned block.
//   kAtlasQuads: RGBO, 64 or 32 bytes (SHADE);
//   kAtlasOcc:   O alone, as float4 (float32 atlas) or four 16-bit values
//                (SHADOW reads only O, Eq. 8);
//   kAtlasCheck: nothing stored (the kernels that read the atlas itself);
// in each the texels are checked: every interior texel is the first texel of
// one footprint.
enum { kAtlasQuads = 0, kAtlasOcc = 1, kAtlasCheck = 2 };
template <int DT>
__device__ __forceinline__ void atlas_footprint(const typename Texel<DT>::raw* __restrict__ atlas, int32_t R, int64_t i,
                                                int what, void* __restrict__ quads, unsigned int* status)
{
    using raw = typename Texel<DT>::raw;
    const int RS = R + 2, RQ = R + 1;
    const int64_t pr = i / (RQ * RQ);
    const int r = (int)(i % (RQ * RQ));
    const int b = r / RQ, a = r % RQ;
    const raw* src = atlas + pr * RS * RS + (int64_t)b * RS + a;
    const raw t0 = src[0];
    if (what == kAtlasOcc && DT == SOP_F32) flag_nonfinite(isfinite(reinterpret_cast<const float4&>(t0).w), status);
    else flag_nonfinite(Texel<DT>::finite(t0), status);
    if (what == kAtlasCheck) return;
    const raw t1 = src[1], t2 = src[RS], t3 = src[RS + 1];
    if (what == kAtlasQuads) {
        raw* dst = reinterpret_cast<raw*>(quads) + 4 * i;
        dst[0] = t0;
        dst[1] = t1;
        dst[2] = t2;
        dst[3] = t3;
    } else if (DT == SOP_F32) {
        const auto w = [](const raw& t) { return reinterpret_cast<const float4&>(t).w; };
        reinterpret_cast<float4*>(quads)[i] = make_float4(w(t0), w(t1), w(t2), w(t3));
    } else {
        // O is the upper half of the second word
        const auto y = [](const raw& t) { return reinterpret_cast<const uint2&>(t).y; };
        reinterpret_cast<uint2*>(quads)[i] = make_uint2((y(t0) >> 16) | (y(t1) & 0xffff0000u),
                                                        (y(t2) >> 16) | (y(t3) & 0xffff0000u));
    }
}

__device__ __forceinline__ double radical_inverse2(uint32_t i) { return (double)__brev(i) * 2.3283064365386963e-10; }

// Local light direction i: the caller's, or the centred Hammersley set's.
__device__ __forceinline__ float3 local_dir(int i, int32_t S, const float* __restrict__ dirs_local)
{
    if (dirs_local) return load3(dirs_local, i);
    const double z = (i + 0.5) / S;
    const double phi = 6.283185307179586476925 * radical_inverse2((uint32_t)i);
    const double s = sqrt(1.0 - z * z);
    return f3((float)(s * cos(phi)), (float)(s * sin(phi)), (float)z);
}

__global__ void dirs_kernel(int32_t S, const float* __restrict__ dirs_local, float4* __restrict__ out4,
                            float* __restrict__ out3)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S) return;
    const float3 d = local_dir(i, S, dirs_local);
    if (out4) out4[i] = make_float4(d.x, d.y, d.z, 0.f);
    if (out3) {
        out3[3 * i] = d.x;
        out3[3 * i + 1] = d.y;
        out3[3 * i + 2] = d.z;
    }
}

// The probe grid and the tables of one query, by block: [0, n_grid) the grid,
// then n_dirs blocks of directions, n_env of environment footprints, and the
// rest of atlas footprints. They are independent of one another, and the
// first, a serial chain, runs beside the others; seven launches before.
struct TablesK {
    const float* probe_pos;
    int32_t P, g_axis;
    ProbeGrid* grid;
    int32_t *cell_start, *cell_cnt;
    int4* entries;
    const float* env;
    int32_t He, We, env_layout;
    float4* envq;
    const void* atlas;
    int32_t R, dtype, what;
    void* quads;
    const float* dirs_in;
    int32_t S, dir_world;
    float4* dirs;
    unsigned n_grid, n_dirs, n_env;
    unsigned int* status;
};

__global__ void __launch_bounds__(kGridThreads) query_tables_kernel(const TablesK k)
{
    __shared__ GridSmem sm;
    unsigned b = blockIdx.x;
    if (b < k.n_grid) {
        probe_grid_build(sm, k.probe_pos, k.P, k.g_axis, k.grid, k.cell_start, k.cell_cnt, k.entries);
        return;
    }
    b -= k.n_grid;
    if (b < k.n_dirs) {
        const int i = b * kGridThreads + threadIdx.x;
        if (i >= k.S) return;
        if (k.dir_world) {
            // importance-sampled (x, y, z, pdf) -> (x, y, z, 1/pdf)
            const float4 d = reinterpret_cast<const float4*>(k.dirs_in)[i];
            k.dirs[i] = make_float4(d.x, d.y, d.z, 1.f / d.w);
        } else {
            const float3 d = local_dir(i, k.S, k.dirs_in);
            k.dirs[i] = make_float4(d.x, d.y, d.z, 0.f);
        }
        return;
    }
    b -= k.n_dirs;
    if (b < k.n_env) {
        const int64_t i = (int64_t)b * kGridThreads + threadIdx.x;
        if (!k.envq) {  // checked only
            if (i < (int64_t)k.He * k.We) {
                const float3 e = load3(k.env, i);
                flag_nonfinite(isfinite(e.x + e.y + e.z), k.status);
            }
        } else if (k.env_layout == SOP_ENV_OCTAHEDRAL) {
            if (i < (int64_t)(k.He + 1) * (k.He + 1)) env_oct_footprint(k.env, k.He, i, k.envq, k.status);
        } else if (i < (int64_t)(k.He + 1) * k.We) {
            env_footprint(k.env, k.He, k.We, i, k.envq, k.status);
        }
        return;
    }
    b -= k.n_env;
    const int64_t i = (int64_t)b * kGridThreads + threadIdx.x;
    if (i >= (int64_t)k.P * (k.R + 1) * (k.R + 1)) return;
    if (k.dtype == SOP_F32)
        atlas_footprint<SOP_F32>(reinterpret_cast<const float4*>(k.atlas), k.R, i, k.what, k.quads, k.status);
    else if (k.dtype == SOP_BF16)
        atlas_footprint<SOP_BF16>(reinterpret_cast<const uint2*>(k.atlas), k.R, i, k.what, k.quads, k.status);
    else atlas_footprint<SOP_F16>(reinterpret_cast<const uint2*>(k.atlas), k.R, i, k.what, k.quads, k.status);
}

// 256-bit read-only global load (sm_100+); p must be 32-byte aligned.
__device__ __forceinline__ void ldg256(const void* p, uint64_t& a, uint64_t& b, uint64_t& c, uint64_t& d)
{
    asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];"
        : "=l"(a), "=l"(b), "=l"(c), "=l"(d)
        : "l"(p));
}
__device__ __forceinline__ float lo32f(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi32f(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }

// Bilinear environment lookup L_dir(w) (z-up equirectangular) from the
// footprint table: three 16-byte loads of one 64-byte slot.
__device__ __forceinline__ float3 env_lookup(const float4* __restrict__ envq, int He, int We, float3 w)
{
    const float th = atan2f(sqrtf(w.x * w.x + w.y * w.y), w.z);
    const float ph = atan2f(w.y, w.x);
    const float s = (ph + kPi) * kInv2Pi * We - 0.5f;
    const float t = th * kInvPi * He - 0.5f;
    const float fs = floorf(s), ft = floorf(t);
    const float a = s - fs, b = t - ft;
    int c0 = (int)fs;
    c0 = c0 < 0 ? c0 + We : c0;
    c0 = min(max(c0, 0), We - 1);
    const int r0 = min(max((int)ft + 1, 0), He);
    const float4* q = envq + 4 * ((int64_t)r0 * We + c0);
    uint64_t x0, x1, x2, x3;
    ldg256(q, x0, x1, x2, x3);
    const float4 q0 = make_float4(lo32f(x0), hi32f(x0), lo32f(x1), hi32f(x1));
    const float4 q1 = make_float4(lo32f(x2), hi32f(x2), lo32f(x3), hi32f(x3));
    const float4 q2 = __ldg(q + 2);
    const float w00 = (1.f - a) * (1.f - b), w01 = a * (1.f - b), w10 = (1.f - a) * b, w11 = a * b;
    return f3(w00 * q0.x + w01 * q0.w + w10 * q1.z + w11 * q2.y, w00 * q0.y + w01 * q1.x + w10 * q1.w + w11 * q2.z,
              w00 * q0.z + w01 * q1.y + w10 * q2.x + w11 * q2.w);
}

// Bilinear lookup of an octahedral environment (Sec. 4.1) at the octahedral
// coordinates uv of the direction (the probe maps' mapping: no atan2), from
// the footprint table that env_oct_footprint wrote.
__device__ __forceinline__ float3 env_oct_lookup(const float4* __restrict__ envq, int H, float2 uv)
{
    const float s = uv.x * H - 0.5f, t = uv.y * H - 0.5f;
    const float fs = floorf(s), ft = floorf(t);
    const float a = s - fs, b = t - ft;
    const int c0 = min(max((int)fs + 1, 0), H), r0 = min(max((int)ft + 1, 0), H);
    const float4* q = envq + 4 * ((int64_t)r0 * (H + 1) + c0);
    uint64_t x0, x1, x2, x3;
    ldg256(q, x0, x1, x2, x3);
    const float4 q0 = make_float4(lo32f(x0), hi32f(x0), lo32f(x1), hi32f(x1));
    const float4 q1 = make_float4(lo32f(x2), hi32f(x2), lo32f(x3), hi32f(x3));
    const float4 q2 = __ldg(q + 2);
    const float w00 = (1.f - a) * (1.f - b), w01 = a * (1.f - b), w10 = (1.f - a) * b, w11 = a * b;
    return f3(w00 * q0.x + w01 * q0.w + w10 * q1.z + w11 * q2.y, w00 * q0.y + w01 * q1.x + w10 * q1.w + w11 * q2.z,
              w00 * q0.z + w01 * q1.y + w10 * q2.x + w11 * q2.w);
}

// One bilinear footprint of the atlas: four texels as float4 (RGB, O).
template <int DT> struct Quad;
template <> struct Quad<SOP_F32> {
    static __device__ __forceinline__ void load(const void* base, int64_t qi, float4& t00, float4& t10, float4& t01,
                                                float4& t11)
    {
        const float4* p = reinterpret_cast<const float4*>(base) + 4 * qi;
        uint64_t a, b, c, d, e, f, g, h;
        ldg256(p, a, b, c, d);
        ldg256(p + 2, e, f, g, h);
        t00 = make_float4(lo32f(a), hi32f(a), lo32f(b), hi32f(b));
        t10 = make_float4(lo32f(c), hi32f(c), lo32f(d), hi32f(d));
        t01 = make_float4(lo32f(e), hi32f(e), lo32f(f), hi32f(f));
        t11 = make_float4(lo32f(g), hi32f(g), lo32f(h), hi32f(h));
    }
};
__device__ __forceinline__ float4 h4(uint32_t x, uint32_t y)
{
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 b4(uint32_t x, uint32_t y)
{
    return make_float4(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u), __uint_as_float(y << 16),
                       __uint_as_float(y & 0xffff0000u));
}
template <> struct Quad<SOP_F16> {
    static __device__ __forceinline__ void load(const void* base, int64_t qi, float4& t00, float4& t10, float4& t01,
                                                float4& t11)
    {
        uint64_t a, b, c, d;
        ldg256(reinterpret_cast<const uint4*>(base) + 2 * qi, a, b, c, d);
        t00 = h4((uint32_t)a, (uint32_t)(a >> 32));
        t10 = h4((uint32_t)b, (uint32_t)(b >> 32));
        t01 = h4((uint32_t)c, (uint32_t)(c >> 32));
        t11 = h4((uint32_t)d, (uint32_t)(d >> 32));
    }
};
template <> struct Quad<SOP_BF16> {
    static __device__ __forceinline__ void load(const void* base, int64_t qi, float4& t00, float4& t10, float4& t01,
                                                float4& t11)
    {
        uint64_t a, b, c, d;
        ldg256(reinterpret_cast<const uint4*>(base) + 2 * qi, a, b, c, d);
        t00 = b4((uint32_t)a, (uint32_t)(a >> 32));
        t10 = b4((uint32_t)b, (uint32_t)(b >> 32));
        t01 = b4((uint32_t)c, (uint32_t)(c >> 32));
        t11 = b4((uint32_t)d, (uint32_t)(d >> 32));
    }
};

// One occlusion footprint: O at (a,b), (a+1,b), (a,b+1), (a+1,b+1).
template <int DT> struct OQuad;
template <> struct OQuad<SOP_F32> {
    static __device__ __forceinline__ float4 load(const void* base, int64_t qi)
    {
        return __ldg(reinterpret_cast<const float4*>(base) + qi);
    }
};
template <> struct OQuad<SOP_F16> {
    static __device__ __forceinline__ float4 load(const void* base, int64_t qi)
    {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(base) + qi);
        return h4(v.x, v.y);
    }
};
template <> struct OQuad<SOP_BF16> {
    static __device__ __forceinline__ float4 load(const void* base, int64_t qi)
    {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(base) + qi);
        return b4(v.x, v.y);
    }
};

// Geometry of one light direction at a point: the world direction (local
// direction l rotated into the frame (t, b, n)), its octahedral footprint
// (offset of the base texel in a probe's stored map) and bilinear weights.
struct DirTerms {
    float3 w;
    float2 uv;
    int off;
    float fu, fv;
    float w00, w10, w01, w11;
};
// footprint part for a world direction w
__device__ __forceinline__ DirTerms footprint_terms(const float3 w, const float Rf, const int R, const int RQ)
{
    DirTerms d;
    d.w = w;
    const float2 uv = oct_encode(d.w);
    d.uv = uv;
    const float s = uv.x * Rf - 0.5f, t = uv.y * Rf - 0.5f;
    const float fi = floorf(s), fj = floorf(t);
    const float fu = s - fi, fv = t - fj;
    const int i0 = min(max((int)fi + 1, 0), R), j0 = min(max((int)fj + 1, 0), R);
    d.off = j0 * RQ + i0;
    d.fu = fu;
    d.fv = fv;
    d.w00 = (1.f - fu) * (1.f - fv);
    d.w10 = fu * (1.f - fv);
    d.w01 = (1.f - fu) * fv;
    d.w11 = fu * fv;
    return d;
}

__device__ __forceinline__ DirTerms dir_terms(const float4 l, const float3 tt, const float3 bb, const float3 n,
                                              const float Rf, const int R, const int RQ)
{
    return footprint_terms(f3(fmaf(l.x, tt.x, fmaf(l.y, bb.x, l.z * n.x)), fmaf(l.x, tt.y, fmaf(l.y, bb.y, l.z * n.y)),
                              fmaf(l.x, tt.z, fmaf(l.y, bb.z, l.z * n.z))),
                           Rf, R, RQ);
}

// Blended occlusion of one direction over a point's K probes (Eq. 5, applied
// to O): each footprint corner is blended over the probes, then the four
// corners are weighted once, O = sum_c w_c sum_k W_k O_k,c.
template <int DT, int KMAX>
__device__ __forceinline__ float shadow_blend(const void* quads, const int32_t* base, const float* W, const int K,
                                              const int off, const float w00, const float w10, const float w01,
                                              const float w11)
{
    float s00 = 0.f, s10 = 0.f, s01 = 0.f, s11 = 0.f;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        if (k < K) {
            const float4 q = OQuad<DT>::load(quads, (int64_t)(base[k] + off));
            s00 = fmaf(W[k], q.x, s00);
            s10 = fmaf(W[k], q.y, s10);
            s01 = fmaf(W[k], q.z, s01);
            s11 = fmaf(W[k], q.w, s11);
        }
    }
    return fmaf(w00, s00, fmaf(w10, s10, fmaf(w01, s01, w11 * s11)));
}

// SHADOW-mode warps whose points share a normal keep per-direction terms in
// shared memory (32 bytes a direction per warp) for S up to this
constexpr int kShadowTab = 128;

struct ShadeK {
    const float *n, *wo, *albedo, *rough, *metal;
    int64_t M;
    const void* rgbo;
    int32_t R, K, S, He, We;
    const float4* envq;
    int32_t env_layout;
    const void* quads;
    const float4* dirs;
    const int32_t* idx;
    const float* w;
    float specular;
    float* out;
    unsigned int* status;  // device status word or NULL
};

// ---------------------------------------------------------------------------
// Query + shade. LANES consecutive threads share one point and split its S
// directions; one warp covers 32/LANES points.
// ---------------------------------------------------------------------------
template <int DT, int KMAX, int MODE>
__global__ void __launch_bounds__(256, 4) shade_kernel(const ShadeK a, const int LANES)
{
    extern __shared__ float4 s_dirs[];
    for (int i = threadIdx.x; i < a.S; i += blockDim.x) s_dirs[i] = a.dirs[i];
    __syncthreads();
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t m = gid / LANES;
    const int sub = (int)(gid % LANES);
    const bool active = m < a.M;
    const int64_t mm = active ? m : 0;

    const float3 nr = load3(a.n, mm);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 n = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    float3 tt, bb;
    onb(n, tt, bb);
    const float3 wo = load3(a.wo, mm);
    const int RQ = a.R + 1;
    int32_t base[KMAX];
    float W[KMAX];
    int32_t ids[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const bool on = k < a.K;
        ids[k] = on ? __ldg(a.idx + mm * a.K + k) : INT32_MAX;
        W[k] = on ? __ldg(a.w + mm * a.K + k) : 0.f;
    }
    // visit the probes in index order: neighbouring points, which share most
    // of their probes, then read the same footprints at the same time
    if (KMAX <= 8)
#pragma unroll
    for (int i = 1; i < KMAX; ++i)
#pragma unroll
        for (int j = KMAX - 1; j >= i; --j) {
            const bool sw = ids[j - 1] > ids[j];
            const int32_t ti = ids[j - 1];
            const float tw = W[j - 1];
            ids[j - 1] = sw ? ids[j] : ids[j - 1];
            W[j - 1] = sw ? W[j] : W[j - 1];
            ids[j] = sw ? ti : ids[j];
            W[j] = sw ? tw : W[j];
        }
#pragma unroll
    for (int k = 0; k < KMAX; ++k) base[k] = (k < a.K) ? ids[k] * RQ * RQ : 0;
    // per-point BRDF constants
    float3 kd, F0;
    float a2 = 0.f, kk = 0.f, specV = 0.f, NdotV = 1.f;
    if (MODE == SOP_MODE_SHADE) {
        const float3 alb = load3(a.albedo, mm);
        const float r = __ldg(a.rough + mm), mt = __ldg(a.metal + mm);
        if (a.status && active && sub == 0 && !isfinite(alb.x + alb.y + alb.z + r + mt + wo.x + wo.y + wo.z))
            atomicOr(a.status, SOP_DEVSTAT_NONFINITE);
        const float dsc = (1.f - mt) * kInvPi;
        kd = f3(dsc * alb.x, dsc * alb.y, dsc * alb.z);
        const float f0d = 0.08f * a.specular * (1.f - mt);
        F0 = f3(f0d + alb.x * mt, f0d + alb.y * mt, f0d + alb.z * mt);
        const float al = r * r;
        a2 = al * al;
        kk = (r + 1.f) * (r + 1.f) * 0.125f;
        NdotV = fmaxf(dot3(n, wo), 1e-4f);
        const float G1V = NdotV / (NdotV * (1.f - kk) + kk);
        specV = G1V / (4.f * NdotV);
    }
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, den0 = 0.f, den1 = 0.f, den2 = 0.f;
    const float Rf = (float)a.R;
    // SHADOW mode, every point of the warp on the same normal (bit for bit; a
    // planar receiver such as a ground plane): their light directions, and so
    // the footprint offsets, bilinear weights and environment terms of every
    // direction, coincide (Eq. 3 rotates one local set by the normal's frame).
    // The lanes then compute those once for the warp into shared memory, and
    // each point only gathers and blends its own probes.
    bool warp_dirs = false;
    if (MODE == SOP_MODE_SHADOW && a.S <= kShadowTab) {
        const unsigned full = 0xffffffffu;
        const unsigned bx = __float_as_uint(nr.x), by = __float_as_uint(nr.y), bz = __float_as_uint(nr.z);
        // every lane takes all three shuffles (no short-circuit: a lane that
        // skipped one would leave the others waiting at it)
        const unsigned x0 = __shfl_sync(full, bx, 0), y0 = __shfl_sync(full, by, 0), z0 = __shfl_sync(full, bz, 0);
        const bool same = (bx == x0) & (by == y0) & (bz == z0);
        warp_dirs = __all_sync(full, same);
    }
    if (MODE == SOP_MODE_SHADOW && warp_dirs) {
        float4* tab = s_dirs + a.S + (threadIdx.x >> 5) * 2 * a.S;
        for (int i = (int)(threadIdx.x & 31); i < a.S; i += 32) {
            const float4 l = s_dirs[i];
            const DirTerms d = dir_terms(l, tt, bb, n, Rf, a.R, RQ);
            const float3 Ld = a.env_layout == SOP_ENV_OCTAHEDRAL ? env_oct_lookup(a.envq, a.He, d.uv)
                                                                 : env_lookup(a.envq, a.He, a.We, d.w);
            const float NdotL = l.z;
            tab[i] = make_float4(__int_as_float(d.off), d.w00, d.w10, d.w01);
            tab[a.S + i] = make_float4(d.w11, Ld.x * NdotL, Ld.y * NdotL, Ld.z * NdotL);
        }
        __syncwarp();
        for (int i = sub; i < a.S; i += LANES) {
            const float4 ta = tab[i], tb = tab[a.S + i];
            const float vis =
                1.f - shadow_blend<DT, KMAX>(a.quads, base, W, a.K, __float_as_int(ta.x), ta.y, ta.z, ta.w, tb.x);
            acc0 = fmaf(tb.y, vis, acc0);
            acc1 = fmaf(tb.z, vis, acc1);
            acc2 = fmaf(tb.w, vis, acc2);
            den0 += tb.y;
            den1 += tb.z;
            den2 += tb.w;
        }
    } else
    for (int i = sub; i < a.S; i += LANES) {
        const float4 l = s_dirs[i];
        const DirTerms d = dir_terms(l, tt, bb, n, Rf, a.R, RQ);
        const float3 w = d.w;
        const int off = d.off;
        const float w00 = d.w00, w10 = d.w10, w01 = d.w01, w11 = d.w11;
        float4 pr = make_float4(0.f, 0.f, 0.f, 0.f);
        if (MODE == SOP_MODE_SHADOW) {
            pr.w = shadow_blend<DT, KMAX>(a.quads, base, W, a.K, off, w00, w10, w01, w11);
        } else
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            if (k < a.K) {
                float4 t00, t10, t01, t11;
                Quad<DT>::load(a.quads, (int64_t)(base[k] + off), t00, t10, t01, t11);
                const float c00 = W[k] * w00, c10 = W[k] * w10, c01 = W[k] * w01, c11 = W[k] * w11;
                pr.x += c00 * t00.x + c10 * t10.x + c01 * t01.x + c11 * t11.x;
                pr.y += c00 * t00.y + c10 * t10.y + c01 * t01.y + c11 * t11.y;
                pr.z += c00 * t00.z + c10 * t10.z + c01 * t01.z + c11 * t11.z;
                pr.w += c00 * t00.w + c10 * t10.w + c01 * t01.w + c11 * t11.w;
            }
        }
        const float3 Ld = a.env_layout == SOP_ENV_OCTAHEDRAL ? env_oct_lookup(a.envq, a.He, d.uv)
                                                             : env_lookup(a.envq, a.He, a.We, w);
        const float NdotL = l.z;
        const float vis = 1.f - pr.w;
        if (MODE == SOP_MODE_SHADE) {
            float3 h = w + wo;
            const float hl2 = dot3(h, h);
            h = hl2 > 1e-30f ? rsqrtf(hl2) * h : n;
            const float NdotH = dot3(n, h), VdotH = dot3(wo, h);
            const float3 cr = cross3(n, h);
            const float sin2 = dot3(cr, cr);
            const float den = NdotH * NdotH * a2 + sin2;
            const float D = __fdividef(a2, kPi * den * den);
            const float spec = __fdividef(D * specV, NdotL * (1.f - kk) + kk);
            const float x1 = 1.f - VdotH, x2 = x1 * x1, fc = x2 * x2 * x1;
            const float f0 = kd.x + spec * (F0.x + (1.f - F0.x) * fc);
            const float f1 = kd.y + spec * (F0.y + (1.f - F0.y) * fc);
            const float f2 = kd.z + spec * (F0.z + (1.f - F0.z) * fc);
            acc0 += f0 * (vis * Ld.x + pr.x) * NdotL;
            acc1 += f1 * (vis * Ld.y + pr.y) * NdotL;
            acc2 += f2 * (vis * Ld.z + pr.z) * NdotL;
        } else {
            // the same terms, in the same order, as the shared-direction path
            const float L0 = Ld.x * NdotL, L1 = Ld.y * NdotL, L2 = Ld.z * NdotL;
            acc0 = fmaf(L0, vis, acc0);
            acc1 = fmaf(L1, vis, acc1);
            acc2 = fmaf(L2, vis, acc2);
            den0 += L0;
            den1 += L1;
            den2 += L2;
        }
    }
    for (int o = LANES / 2; o > 0; o >>= 1) {
        acc0 += __shfl_xor_sync(0xffffffffu, acc0, o);
        acc1 += __shfl_xor_sync(0xffffffffu, acc1, o);
        acc2 += __shfl_xor_sync(0xffffffffu, acc2, o);
        if (MODE == SOP_MODE_SHADOW) {
            den0 += __shfl_xor_sync(0xffffffffu, den0, o);
            den1 += __shfl_xor_sync(0xffffffffu, den1, o);
            den2 += __shfl_xor_sync(0xffffffffu, den2, o);
        }
    }
    if (active && sub == 0) {
        float* o = a.out + 3 * m;
        if (MODE == SOP_MODE_SHADE) {
            const float sc = 2.f * kPi / (float)a.S;
            o[0] = sc * acc0;
            o[1] = sc * acc1;
            o[2] = sc * acc2;
        } else {
            o[0] = den0 < 1e-20f ? 1.f : acc0 / den0;
            o[1] = den1 < 1e-20f ? 1.f : acc1 / den1;
            o[2] = den2 < 1e-20f ? 1.f : acc2 / den2;
        }
    }
}

// ---------------------------------------------------------------------------
// SHADOW mode, large calls: one thread per point.
//
// The shadow ratio is sum_i L_i cos_i (1 - O(w_i)) / sum_i L_i cos_i with O =
// sum_k W_k O_k (Eq. 5 applied to O), so the sum over directions can be taken
// per probe first: V_k = sum_i L_i cos_i (1 - O_k(w_i)), and over the probes
// what is visible, num = sum_k W_k V_k, and what is hidden, hid = sum_k W_k (den
// - V_k): the ratio is num / (num + hid), taken from the smaller of the two, so
// that what is left of a hidden light is no difference of large sums and a
// point that nothing hides is exactly 1. (The weights' sum is 1 but for its
// rounding, which cancels.) V_k depends on the point only through its normal.
// Where the points of
// a warp share one normal bit for bit (a planar receiver such as a ground
// plane: their directions, footprints and environment terms coincide), the
// warp takes each of its distinct probes once, the lanes over the directions,
// and the 32 points combine the results: a few probes times S footprints a
// warp instead of 32 K S. Neighbouring points share nearly all their probes
// (about 10 distinct of 256); a warp with more than kShadowProbes of them, or
// with several normals, blends per point and direction as shade_kernel does.
// Bound: the reads of normals, indices and weights, then issue. 2,051,693
// ground points, K = 8, S = 64, 16-bit atlas: 716 -> 262 us (normals equal bit for
// bit, as an analytic plane's are; normals of a traced G-buffer differ in their
// last bits from pixel to pixel: the whole call 1,945 -> 1,739 us with 1e-7 of
// noise, most of it from the search).
// ---------------------------------------------------------------------------
constexpr int kShadowProbes = 32;
// Whole calls, us (lanes / warp): 16-bit atlas, S 64: 32,768 points 163 / 208,
// 131,072: 208 / 217 (on a ground), 248 / 260 (on an object: mixed normals),
// float32 on an object 284 / 274; 2,051,693 on a ground: 1,240 / 776. A warp's
// few serial steps do not fill the machine below.
constexpr int64_t kShadowWarpPoints = 262144;
// Up to 16 probes a point: 32 spill (1,000,000 ground points, K 32, whole call:
// 3,614 us in lanes, 4,025 here; K 16: 1,328 / 955).
constexpr int kShadowWarpK = 16;

// Ratio of one point by blending per direction, LANES threads a point.
template <int DT, int KMAX, int LANES>
__device__ __forceinline__ void shadow_point(const ShadeK& a, const float4* __restrict__ s_dirs, const int64_t m,
                                             const int sub, const bool active)
{
    const int64_t mm = active ? m : 0;
    const float3 nr = load3(a.n, mm);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 n = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    float3 tt, bb;
    onb(n, tt, bb);
    const int RQ = a.R + 1;
    int32_t base[KMAX];
    float W[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const bool on = k < a.K;
        base[k] = on ? __ldg(a.idx + mm * a.K + k) * RQ * RQ : 0;
        W[k] = on ? __ldg(a.w + mm * a.K + k) : 0.f;
    }
    float acc[3] = {0.f, 0.f, 0.f}, den[3] = {0.f, 0.f, 0.f};
    const float Rf = (float)a.R;
    for (int i = sub; i < a.S; i += LANES) {
        const float4 l = s_dirs[i];
        const DirTerms d = dir_terms(l, tt, bb, n, Rf, a.R, RQ);
        const float vis = 1.f - shadow_blend<DT, KMAX>(a.quads, base, W, a.K, d.off, d.w00, d.w10, d.w01, d.w11);
        const float3 Ld = a.env_layout == SOP_ENV_OCTAHEDRAL ? env_oct_lookup(a.envq, a.He, d.uv)
                                                             : env_lookup(a.envq, a.He, a.We, d.w);
        const float L[3] = {Ld.x * l.z, Ld.y * l.z, Ld.z * l.z};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc[c] = fmaf(L[c], vis, acc[c]);
            den[c] += L[c];
        }
    }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
            den[c] += __shfl_xor_sync(0xffffffffu, den[c], o);
        }
    if (active && sub == 0)
#pragma unroll
        for (int c = 0; c < 3; ++c) a.out[3 * m + c] = den[c] < 1e-20f ? 1.f : acc[c] / den[c];
}

// LANES: threads a point of the warps without a common normal (shade_lanes)
template <int DT, int KMAX, int LANES>
__global__ void __launch_bounds__(256, 4) shadow_warp_kernel(const ShadeK a)
{
    extern __shared__ float4 s_dirs[];
    for (int i = threadIdx.x; i < a.S; i += blockDim.x) s_dirs[i] = a.dirs[i];
    __syncthreads();
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t m0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~(int64_t)31;  // the warp's first point
    if (m0 >= a.M) return;
    const int64_t m = m0 + lane;
    const bool active = m < a.M;
    const int64_t mm = active ? m : a.M - 1;
    const float3 nr = load3(a.n, mm);
    // every lane takes all three shuffles (no short-circuit)
    const unsigned bx = __float_as_uint(nr.x), by = __float_as_uint(nr.y), bz = __float_as_uint(nr.z);
    const unsigned x0 = __shfl_sync(full, bx, 0), y0 = __shfl_sync(full, by, 0), z0 = __shfl_sync(full, bz, 0);
    bool shared = __all_sync(full, (bx == x0) & (by == y0) & (bz == z0));
    const int RQ = a.R + 1;
    int32_t id[KMAX];
    float W[KMAX];
    if (shared) {
        // the warp's distinct probes, ascending, one a lane
        int32_t mine = 0, last = -1;
        int n = 0;
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            const bool on = k < a.K;
            id[k] = on ? __ldg(a.idx + mm * a.K + k) : INT32_MAX;
            W[k] = on ? __ldg(a.w + mm * a.K + k) : 0.f;
        }
        for (;; ++n) {
            int32_t next = INT32_MAX;
#pragma unroll
            for (int k = 0; k < KMAX; ++k) next = min(next, id[k] > last ? id[k] : INT32_MAX);
            next = __reduce_min_sync(full, next);
            if (next == INT32_MAX || n == kShadowProbes) {
                shared = next == INT32_MAX;
                break;
            }
            if (lane == n) mine = next;
            last = next;
        }
        if (shared) {
            const float nl = sqrtf(dot3(nr, nr));
            const float3 nn = f3(nr.x / nl, nr.y / nl, nr.z / nl);
            float3 tt, bb;
            onb(nn, tt, bb);
            // this lane's directions: footprint, weights, environment times cos
            constexpr int NR = kShadowTab / 32;
            int off[NR];
            float fu[NR], fv[NR], L[NR][3], den[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int i = r * 32 + lane;
                off[r] = -1;
                if (i < a.S) {
                    const float4 l = s_dirs[i];
                    const DirTerms d = dir_terms(l, tt, bb, nn, (float)a.R, a.R, RQ);
                    const float3 Ld = a.env_layout == SOP_ENV_OCTAHEDRAL ? env_oct_lookup(a.envq, a.He, d.uv)
                                                                         : env_lookup(a.envq, a.He, a.We, d.w);
                    off[r] = d.off;
                    fu[r] = d.fu;
                    fv[r] = d.fv;
                    L[r][0] = Ld.x * l.z;
                    L[r][1] = Ld.y * l.z;
                    L[r][2] = Ld.z * l.z;
#pragma unroll
                    for (int c = 0; c < 3; ++c) den[c] += L[r][c];
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) den[c] += __shfl_xor_sync(full, den[c], o);
            // two probes a step: their loads overlap, and the sums over the
            // lanes go on in one half of the warp each (in the order of den's,
            // so that a probe that hides nothing has V = den)
            float num[3] = {0.f, 0.f, 0.f}, hid[3] = {0.f, 0.f, 0.f};
            const bool lower = lane < 16;
            for (int u = 0; u < n; u += 2) {
                int32_t p[2];
                float V[2][3], w[2] = {0.f, 0.f};
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    p[j] = __shfl_sync(full, mine, min(u + j, n - 1));
#pragma unroll
                    for (int c = 0; c < 3; ++c) V[j][c] = 0.f;
                }
#pragma unroll
                for (int r = 0; r < NR; ++r)
                    if (off[r] >= 0) {
                        const float4 qa = OQuad<DT>::load(a.quads, (int64_t)(p[0] * RQ * RQ + off[r]));
                        const float4 qb = OQuad<DT>::load(a.quads, (int64_t)(p[1] * RQ * RQ + off[r]));
                        const float la = fmaf(fu[r], qa.y - qa.x, qa.x), ha = fmaf(fu[r], qa.w - qa.z, qa.z);
                        const float lb = fmaf(fu[r], qb.y - qb.x, qb.x), hb = fmaf(fu[r], qb.w - qb.z, qb.z);
                        const float va = 1.f - fmaf(fv[r], ha - la, la), vb = 1.f - fmaf(fv[r], hb - lb, lb);
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            V[0][c] = fmaf(L[r][c], va, V[0][c]);
                            V[1][c] = fmaf(L[r][c], vb, V[1][c]);
                        }
                    }
#pragma unroll
                for (int k = 0; k < KMAX; ++k) {
                    w[0] += id[k] == p[0] ? W[k] : 0.f;
                    w[1] += id[k] == p[1] ? W[k] : 0.f;
                }
                if (u + 1 == n) w[1] = 0.f;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float v = (lower ? V[0][c] : V[1][c]) + __shfl_xor_sync(full, lower ? V[1][c] : V[0][c], 16);
#pragma unroll
                    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
                    const float x = __shfl_xor_sync(full, v, 16), va = lower ? v : x, vb = lower ? x : v;
                    if (w[0] != 0.f) {
                        num[c] = fmaf(w[0], va, num[c]);
                        hid[c] = fmaf(w[0], den[c] - va, hid[c]);
                    }
                    if (w[1] != 0.f) {
                        num[c] = fmaf(w[1], vb, num[c]);
                        hid[c] = fmaf(w[1], den[c] - vb, hid[c]);
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                // (no probe found: both sums are 0, nothing hides the point)
                const float sum = num[c] + hid[c];
                const float ratio = hid[c] <= num[c] ? 1.f - (hid[c] != 0.f ? hid[c] / sum : 0.f) : num[c] / sum;
                if (active) a.out[3 * m + c] = den[c] < 1e-20f ? 1.f : ratio;
            }
            return;
        }
    }
    for (int j = 0; j < LANES; ++j) {
        const int64_t mj = m0 + j * (32 / LANES) + lane / LANES;
        shadow_point<DT, KMAX, LANES>(a, s_dirs, mj, lane % LANES, mj < a.M);
    }
}

// ---------------------------------------------------------------------------
// Query + shade, SHADE mode, one warp per point (point_blend.cuh): lanes
// share the directions, 32 a round. NR: rounds whose footprints stay in
// registers between the marking and the shading (S <= 32 NR), or 0: any S,
// computed twice. Bound: L1 and shared memory (92% of their throughput): the
// blended texels (20 KB a point at R = 16, K = 8), four of them a direction
// from shared memory, the environment's gathers. 418,111 points, K = 8,
// S = 128: 1,717 -> 1,400 us against shade_kernel.
// ---------------------------------------------------------------------------
template <int DT, int KMAX, int NR>
__global__ void __launch_bounds__(kPointWarps * 32, 4) shade_point_kernel(const ShadeK a)
{
    using TX = Texel<DT>;
    extern __shared__ float4 s_dirs[];
    for (int i = threadIdx.x; i < a.S; i += blockDim.x) s_dirs[i] = a.dirs[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t m = (int64_t)blockIdx.x * kPointWarps + warp;
    if (m >= a.M) return;
    const PointSmem sm = point_smem(reinterpret_cast<char*>(s_dirs + a.S) + warp * point_smem_bytes(a.R), a.R);
    const int RS = a.R + 2, words = point_words(a.R);
    const uint32_t RS2 = (uint32_t)(RS * RS);
    const float Rf = (float)a.R;
    for (int w = lane; w <= words; w += 32) sm.mark[w] = 0u;
    const float3 nr = load3(a.n, m);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 n = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    float3 tt, bb;
    onb(n, tt, bb);
    const auto world = [&](const float4 l) {
        return f3(fmaf(l.x, tt.x, fmaf(l.y, bb.x, l.z * n.x)), fmaf(l.x, tt.y, fmaf(l.y, bb.y, l.z * n.y)),
                  fmaf(l.x, tt.z, fmaf(l.y, bb.z, l.z * n.z)));
    };
    __syncwarp();
    Foot ft[NR > 0 ? NR : 1];
    if (NR > 0) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int i = r * 32 + lane;
            ft[r] = oct_foot(world(s_dirs[min(i, a.S - 1)]), Rf, a.R);
            if (i < a.S) point_mark(sm, ft[r].off, RS);
        }
    } else {
        for (int i = lane; i < a.S; i += 32) point_mark(sm, oct_foot(world(s_dirs[i]), Rf, a.R).off, RS);
    }
    __syncwarp();
    const int nt = point_list(sm, words, lane);
    // the point's probes and weights
    uint32_t base[KMAX];
    float W[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const bool on = k < a.K;
        base[k] = on ? (uint32_t)__ldg(a.idx + m * a.K + k) * RS2 : 0u;
        W[k] = on ? __ldg(a.w + m * a.K + k) : 0.f;
    }
    __syncwarp();
    const typename TX::raw* atlas = reinterpret_cast<const typename TX::raw*>(a.rgbo);
    for (int j = lane; j < nt; j += 32) {
        const uint32_t t = sm.list[j];
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < KMAX; ++k)
            if (k < a.K) {
                const float4 x = TX::load(atlas + (base[k] + t));
                v.x = fmaf(W[k], x.x, v.x);
                v.y = fmaf(W[k], x.y, v.y);
                v.z = fmaf(W[k], x.z, v.z);
                v.w = fmaf(W[k], x.w, v.w);
            }
        sm.map[t] = v;
    }
    __syncwarp();
    const float3 wo = load3(a.wo, m);
    const float3 alb = load3(a.albedo, m);
    const float rr = __ldg(a.rough + m), mt = __ldg(a.metal + m);
    if (a.status && lane == 0 && !isfinite(alb.x + alb.y + alb.z + rr + mt + wo.x + wo.y + wo.z))
        atomicOr(a.status, SOP_DEVSTAT_NONFINITE);
    const float dsc = (1.f - mt) * kInvPi;
    const float3 kd = f3(dsc * alb.x, dsc * alb.y, dsc * alb.z);
    const float f0d = 0.08f * a.specular * (1.f - mt);
    const float3 F0 = f3(f0d + alb.x * mt, f0d + alb.y * mt, f0d + alb.z * mt);
    const float al = rr * rr, a2 = al * al, kk = (rr + 1.f) * (rr + 1.f) * 0.125f;
    const float NdotV = fmaxf(dot3(n, wo), 1e-4f);
    const float G1V = NdotV / (NdotV * (1.f - kk) + kk);
    const float specV = G1V / (4.f * NdotV);
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f;
    const auto shade = [&](const float4 l, const Foot f) {
        const float3 w = world(l);
        const float3 Ld = a.env_layout == SOP_ENV_OCTAHEDRAL ? env_oct_lookup(a.envq, a.He, oct_encode(w))
                                                             : env_lookup(a.envq, a.He, a.We, w);
        const float4 t00 = sm.map[f.off], t10 = sm.map[f.off + 1], t01 = sm.map[f.off + RS], t11 = sm.map[f.off + RS + 1];
        const float w00 = (1.f - f.fu) * (1.f - f.fv), w10 = f.fu * (1.f - f.fv), w01 = (1.f - f.fu) * f.fv, w11 = f.fu * f.fv;
        const float3 L = f3(fmaf(w00, t00.x, fmaf(w10, t10.x, fmaf(w01, t01.x, w11 * t11.x))),
                            fmaf(w00, t00.y, fmaf(w10, t10.y, fmaf(w01, t01.y, w11 * t11.y))),
                            fmaf(w00, t00.z, fmaf(w10, t10.z, fmaf(w01, t01.z, w11 * t11.z))));
        const float O = fmaf(w00, t00.w, fmaf(w10, t10.w, fmaf(w01, t01.w, w11 * t11.w)));
        const float vis = 1.f - O, NdotL = l.z;
        float3 h = w + wo;
        const float hl2 = dot3(h, h);
        h = hl2 > 1e-30f ? rsqrtf(hl2) * h : n;
        const float NdotH = dot3(n, h), VdotH = dot3(wo, h);
        const float3 cr = cross3(n, h);
        const float sin2 = dot3(cr, cr);
        const float den = NdotH * NdotH * a2 + sin2;
        const float D = __fdividef(a2, kPi * den * den);
        const float spec = __fdividef(D * specV, NdotL * (1.f - kk) + kk);
        const float x1 = 1.f - VdotH, x2 = x1 * x1, fc = x2 * x2 * x1;
        acc0 += (kd.x + spec * (F0.x + (1.f - F0.x) * fc)) * (vis * Ld.x + L.x) * NdotL;
        acc1 += (kd.y + spec * (F0.y + (1.f - F0.y) * fc)) * (vis * Ld.y + L.y) * NdotL;
        acc2 += (kd.z + spec * (F0.z + (1.f - F0.z) * fc)) * (vis * Ld.z + L.z) * NdotL;
    };
    if (NR > 0) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (r * 32 + lane < a.S) shade(s_dirs[r * 32 + lane], ft[r]);
    } else {
        for (int i = lane; i < a.S; i += 32) {
            const float4 l = s_dirs[i];
            shade(l, oct_foot(world(l), Rf, a.R));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc0 += __shfl_xor_sync(0xffffffffu, acc0, o);
        acc1 += __shfl_xor_sync(0xffffffffu, acc1, o);
        acc2 += __shfl_xor_sync(0xffffffffu, acc2, o);
    }
    if (lane < 3) {
        const float sc = 2.f * kPi / (float)a.S;
        a.out[3 * m + lane] = sc * (lane == 0 ? acc0 : (lane == 1 ? acc1 : acc2));
    }
}

// ---------------------------------------------------------------------------
// Query + shade over importance-sampled world directions (Sec. 4.2): the S
// directions, their octahedral footprints, bilinear weights, environment
// radiance and 1/pdf are the same for every point, so each CTA tabulates
// them once in shared memory (48 bytes a direction). Per point and direction
// there remain the horizon test, the gather of the K probe footprints and,
// in SHADE mode, the BRDF; terms are weighted by 1/pdf and the estimate is
// their sum over the directions above the horizon, divided by S.
// ---------------------------------------------------------------------------
template <int DT, int KMAX, int MODE>
__global__ void __launch_bounds__(256, 4) shade_world_kernel(const ShadeK a, const int LANES)
{
    extern __shared__ float4 s_tab[];  // [S][3]: (w, 1/pdf), (L_dir, off), (w00, w10, w01, w11)
    const float Rf = (float)a.R;
    const int RQ = a.R + 1;
    for (int i = threadIdx.x; i < a.S; i += blockDim.x) {
        const float4 l = a.dirs[i];
        const float3 w = f3(l.x, l.y, l.z);
        const DirTerms d = footprint_terms(w, Rf, a.R, RQ);
        const float3 Ld = a.env_layout == SOP_ENV_OCTAHEDRAL ? env_oct_lookup(a.envq, a.He, d.uv)
                                                             : env_lookup(a.envq, a.He, a.We, w);
        s_tab[3 * i] = l;
        s_tab[3 * i + 1] = make_float4(Ld.x, Ld.y, Ld.z, __int_as_float(d.off));
        s_tab[3 * i + 2] = make_float4(d.w00, d.w10, d.w01, d.w11);
    }
    __syncthreads();
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t m = gid / LANES;
    const int sub = (int)(gid % LANES);
    const bool active = m < a.M;
    const int64_t mm = active ? m : 0;
    const float3 nr = load3(a.n, mm);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 n = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    const float3 wo = load3(a.wo, mm);
    int32_t base[KMAX];
    float W[KMAX];
    int32_t ids[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const bool on = k < a.K;
        ids[k] = on ? __ldg(a.idx + mm * a.K + k) : INT32_MAX;
        W[k] = on ? __ldg(a.w + mm * a.K + k) : 0.f;
    }
    if (KMAX <= 8)
#pragma unroll
    for (int i = 1; i < KMAX; ++i)
#pragma unroll
        for (int j = KMAX - 1; j >= i; --j) {
            const bool sw = ids[j - 1] > ids[j];
            const int32_t ti = ids[j - 1];
            const float tw = W[j - 1];
            ids[j - 1] = sw ? ids[j] : ids[j - 1];
            W[j - 1] = sw ? W[j] : W[j - 1];
            ids[j] = sw ? ti : ids[j];
            W[j] = sw ? tw : W[j];
        }
#pragma unroll
    for (int k = 0; k < KMAX; ++k) base[k] = (k < a.K) ? ids[k] * RQ * RQ : 0;
    float3 kd, F0;
    float a2 = 0.f, kk = 0.f, specV = 0.f, NdotV = 1.f;
    if (MODE == SOP_MODE_SHADE) {
        const float3 alb = load3(a.albedo, mm);
        const float r = __ldg(a.rough + mm), mt = __ldg(a.metal + mm);
        if (a.status && active && sub == 0 && !isfinite(alb.x + alb.y + alb.z + r + mt + wo.x + wo.y + wo.z))
            atomicOr(a.status, SOP_DEVSTAT_NONFINITE);
        const float dsc = (1.f - mt) * kInvPi;
        kd = f3(dsc * alb.x, dsc * alb.y, dsc * alb.z);
        const float f0d = 0.08f * a.specular * (1.f - mt);
        F0 = f3(f0d + alb.x * mt, f0d + alb.y * mt, f0d + alb.z * mt);
        const float al = r * r;
        a2 = al * al;
        kk = (r + 1.f) * (r + 1.f) * 0.125f;
        NdotV = fmaxf(dot3(n, wo), 1e-4f);
        const float G1V = NdotV / (NdotV * (1.f - kk) + kk);
        specV = G1V / (4.f * NdotV);
    }
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, den0 = 0.f, den1 = 0.f, den2 = 0.f;
    for (int i = sub; i < a.S; i += LANES) {
        const float4 ta = s_tab[3 * i], tb = s_tab[3 * i + 1], tc = s_tab[3 * i + 2];
        const float3 w = f3(ta.x, ta.y, ta.z);
        const float NdotL = dot3(n, w);
        if (!(NdotL > 0.f)) continue;  // below the horizon: no contribution
        const int off = __float_as_int(tb.w);
        if (MODE == SOP_MODE_SHADOW) {
            const float vis = 1.f - shadow_blend<DT, KMAX>(a.quads, base, W, a.K, off, tc.x, tc.y, tc.z, tc.w);
            const float c = NdotL * ta.w;
            const float L0 = tb.x * c, L1 = tb.y * c, L2 = tb.z * c;
            acc0 = fmaf(L0, vis, acc0);
            acc1 = fmaf(L1, vis, acc1);
            acc2 = fmaf(L2, vis, acc2);
            den0 += L0;
            den1 += L1;
            den2 += L2;
        } else {
            float4 pr = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < KMAX; ++k) {
                if (k < a.K) {
                    float4 t00, t10, t01, t11;
                    Quad<DT>::load(a.quads, (int64_t)(base[k] + off), t00, t10, t01, t11);
                    const float c00 = W[k] * tc.x, c10 = W[k] * tc.y, c01 = W[k] * tc.z, c11 = W[k] * tc.w;
                    pr.x += c00 * t00.x + c10 * t10.x + c01 * t01.x + c11 * t11.x;
                    pr.y += c00 * t00.y + c10 * t10.y + c01 * t01.y + c11 * t11.y;
                    pr.z += c00 * t00.z + c10 * t10.z + c01 * t01.z + c11 * t11.z;
                    pr.w += c00 * t00.w + c10 * t10.w + c01 * t01.w + c11 * t11.w;
                }
            }
            const float vis = 1.f - pr.w;
            float3 h = w + wo;
            const float hl2 = dot3(h, h);
            h = hl2 > 1e-30f ? rsqrtf(hl2) * h : n;
            const float NdotH = dot3(n, h), VdotH = dot3(wo, h);
            const float3 cr = cross3(n, h);
            const float sin2 = dot3(cr, cr);
            const float den = NdotH * NdotH * a2 + sin2;
            const float D = __fdividef(a2, kPi * den * den);
            const float spec = __fdividef(D * specV, NdotL * (1.f - kk) + kk);
            const float x1 = 1.f - VdotH, x2 = x1 * x1, fc = x2 * x2 * x1;
            const float f0 = kd.x + spec * (F0.x + (1.f - F0.x) * fc);
            const float f1 = kd.y + spec * (F0.y + (1.f - F0.y) * fc);
            const float f2 = kd.z + spec * (F0.z + (1.f - F0.z) * fc);
            const float c = NdotL * ta.w;
            acc0 += f0 * (vis * tb.x + pr.x) * c;
            acc1 += f1 * (vis * tb.y + pr.y) * c;
            acc2 += f2 * (vis * tb.z + pr.z) * c;
        }
    }
    for (int o = LANES / 2; o > 0; o >>= 1) {
        acc0 += __shfl_xor_sync(0xffffffffu, acc0, o);
        acc1 += __shfl_xor_sync(0xffffffffu, acc1, o);
        acc2 += __shfl_xor_sync(0xffffffffu, acc2, o);
        if (MODE == SOP_MODE_SHADOW) {
            den0 += __shfl_xor_sync(0xffffffffu, den0, o);
            den1 += __shfl_xor_sync(0xffffffffu, den1, o);
            den2 += __shfl_xor_sync(0xffffffffu, den2, o);
        }
    }
    if (active && sub == 0) {
        float* o = a.out + 3 * m;
        if (MODE == SOP_MODE_SHADE) {
            const float sc = 1.f / (float)a.S;
            o[0] = sc * acc0;
            o[1] = sc * acc1;
            o[2] = sc * acc2;
        } else {
            o[0] = den0 < 1e-20f ? 1.f : acc0 / den0;
            o[1] = den1 < 1e-20f ? 1.f : acc1 / den1;
            o[2] = den2 < 1e-20f ? 1.f : acc2 / den2;
        }
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
cudaError_t launch_hammersley(int32_t S, float* out3, cudaStream_t s)
{
    dirs_kernel<<<(S + 127) / 128, 128, 0, s>>>(S, nullptr, nullptr, out3);
    return cudaGetLastError();
}

// Up to this many probes a warp a point takes all of them, without a grid.
constexpr int32_t kKnnAllProbes = 256;
// Up to this many points a warp a point; above, a thread a point, which
// issues fewer instructions in all where neighbouring points lie together.
// Whole calls with one light direction, us (thread / warp): 1,000 points 109 /
// 69, 8,191: 105 / 77, 32,768: 119 / 126 in pixel order, 128 / 126 at random,
// 65,536: 136 / 193, 170 / 194.
constexpr int64_t kKnnWarpPoints = 24576;

static bool knn_needs_grid(int32_t P, int64_t M) { return M > kKnnWarpPoints || P > kKnnAllProbes; }

static cudaError_t launch_knn(const KnnK& k, cudaStream_t s)
{
    if (k.M <= kKnnWarpPoints) {
        knn_warp_kernel<<<(unsigned)((k.M + kKnnWarps - 1) / kKnnWarps), kKnnWarps * 32, 0, s>>>(k);
        return cudaGetLastError();
    }
    const int bs = 128;
    const unsigned nb = (unsigned)((k.M + bs - 1) / bs);
    int id_bits = 1;  // of a probe index
    while (id_bits < 31 && ((int64_t)1 << id_bits) < k.P) ++id_bits;
#define SOP_KNN(KM)                                                                                                    \
    knn_kernel<KM><<<nb, bs, 0, s>>>(k.x, k.nrm, k.M, k.K, id_bits, k.snap_key, k.r2_key, k.grid, k.cell_start, k.entries,      \
                                     k.probe_pos, k.ws_idx, k.ws_w, k.user_idx, k.user_w, k.status)
    if (k.K <= 4) SOP_KNN(4);
    else if (k.K <= 8) SOP_KNN(8);
    else if (k.K <= 16) SOP_KNN(16);
    else SOP_KNN(32);
#undef SOP_KNN
    return cudaGetLastError();
}

static bool shade_by_point(const QueryArgs& a);

cudaError_t launch_query_prep(const QueryArgs& a, const QueryLayout& L, char* ws, bool backward, cudaStream_t s)
{
    const auto blocks = [](int64_t n) { return (unsigned)((n + kGridThreads - 1) / kGridThreads); };
    const bool grid = a.M > 0 && knn_needs_grid(a.P, a.M);
    TablesK t;
    t.probe_pos = a.probe_pos;
    t.P = a.P;
    t.g_axis = L.g_axis;
    t.grid = reinterpret_cast<ProbeGrid*>(ws + L.grid_hdr);
    t.cell_start = reinterpret_cast<int32_t*>(ws + L.cell_start);
    t.cell_cnt = reinterpret_cast<int32_t*>(ws + L.cell_cnt);
    t.entries = reinterpret_cast<int4*>(ws + L.entries);
    t.env = a.env;
    t.He = a.He;
    t.We = a.We;
    t.env_layout = a.env_layout;
    t.envq = backward ? nullptr : reinterpret_cast<float4*>(ws + L.envq);  // the adjoint reads the environment itself
    t.atlas = a.rgbo;
    t.R = a.R;
    t.dtype = a.rgbo_dtype;
    t.what = backward || shade_by_point(a) ? kAtlasCheck : (a.mode == SOP_MODE_SHADOW ? kAtlasOcc : kAtlasQuads);
    t.quads = ws + L.quads;
    t.dirs_in = a.dirs_local;
    t.S = a.S;
    t.dir_world = a.dir_world;
    t.dirs = reinterpret_cast<float4*>(ws + L.dirs);
    t.status = status_word();
    t.n_grid = grid ? 1u : 0u;
    t.n_dirs = blocks(a.S);
    t.n_env = blocks(!t.envq ? (int64_t)a.He * a.We
                             : (int64_t)(a.He + 1) * (a.env_layout == SOP_ENV_OCTAHEDRAL ? a.He + 1 : a.We));
    const int64_t n_atlas = (int64_t)a.P * (a.R + 1) * (a.R + 1);
    query_tables_kernel<<<t.n_grid + t.n_dirs + t.n_env + blocks(n_atlas), kGridThreads, 0, s>>>(t);
    if (a.M == 0) return cudaGetLastError();
    KnnK k;
    k.x = a.x;
    k.nrm = a.n;
    k.M = a.M;
    k.K = a.K;
    k.P = a.P;
    k.snap_key = a.snap_key;
    k.r2_key = a.r2_key;
    k.grid = t.grid;
    k.cell_start = t.cell_start;
    k.entries = grid ? t.entries : nullptr;
    k.probe_pos = a.probe_pos;
    k.ws_idx = reinterpret_cast<int32_t*>(ws + L.idx);
    k.ws_w = reinterpret_cast<float*>(ws + L.w);
    k.user_idx = a.out_idx;
    k.user_w = a.out_w;
    k.status = t.status;
    return launch_knn(k, s);
}

template <int DT, int KMAX, int MODE>
static cudaError_t shade_launch(const ShadeK& k, int LANES, cudaStream_t s)
{
    const int bs = 256;
    const int64_t threads = k.M * LANES;
    const unsigned nb = (unsigned)((threads + bs - 1) / bs);
    size_t smem = sizeof(float4) * (size_t)k.S;
    // per-warp direction tables of the shared-normal SHADOW path (8 warps)
    if (MODE == SOP_MODE_SHADOW && k.S <= kShadowTab) smem += (size_t)(bs / 32) * 2 * sizeof(float4) * k.S;
    auto fn = shade_kernel<DT, KMAX, MODE>;
    if (const cudaError_t e = allow_smem(fn, smem); e != cudaSuccess) return e;
    fn<<<nb, bs, smem, s>>>(k, LANES);
    return cudaGetLastError();
}

// Threads per shading point (they split the S directions).
// Measured on GB300, object workload: one thread per point for a float32
// atlas, two for 16-bit atlases; small point sets (the composition frame's
// 21,907 object pixels) take more lanes per point, up to 8, until the launch
// has about two waves of threads on the 152 SMs.
static int shade_lanes(int dtype, int64_t M)
{
    int l = dtype == SOP_F32 ? 1 : 2;
    while (l < 8 && M * l < (int64_t)2 * 152 * 1024) l *= 2;
    return l;
}

template <int DT, int KMAX, int MODE>
static cudaError_t shade_dispatch(const ShadeK& k, cudaStream_t s)
{
    return shade_launch<DT, KMAX, MODE>(k, shade_lanes(DT, k.M), s);
}

template <int DT, int KMAX, int NR>
static cudaError_t shade_point_launch(const ShadeK& k, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * (size_t)k.S + kPointWarps * point_smem_bytes(k.R);
    auto fn = shade_point_kernel<DT, KMAX, NR>;
    if (const cudaError_t e = allow_smem(fn, smem); e != cudaSuccess) return e;
    fn<<<(unsigned)((k.M + kPointWarps - 1) / kPointWarps), kPointWarps * 32, smem, s>>>(k);
    return cudaGetLastError();
}

template <int DT>
static cudaError_t shade_point_k(const ShadeK& k, cudaStream_t s)
{
    if (k.K <= 4) return k.S <= 128 ? shade_point_launch<DT, 4, 4>(k, s) : shade_point_launch<DT, 4, 0>(k, s);
    if (k.K <= 8) return k.S <= 128 ? shade_point_launch<DT, 8, 4>(k, s) : shade_point_launch<DT, 8, 0>(k, s);
    if (k.K <= 16) return k.S <= 128 ? shade_point_launch<DT, 16, 4>(k, s) : shade_point_launch<DT, 16, 0>(k, s);
    return k.S <= 128 ? shade_point_launch<DT, 32, 4>(k, s) : shade_point_launch<DT, 32, 0>(k, s);
}

// Which SHADE kernel: a warp a point pays for the texels that its directions
// touch ((R+2)^2 stored, about half of them) and a fixed amount, then little a
// direction; a thread a point (or a few lanes) pays K footprints a direction.
// Measured on views, us a call (lanes / warp). 418,111 points: float32, R 16,
// K 8: S 128 1,998 / 1,683, S 64 1,153 / 1,305; K 4, S 128 1,116 / 1,335; R 8,
// K 8: S 128 1,938 / 1,423, S 32 697 / 902; R 24, S 128 2,041 / 2,939; 16 bits,
// R 16, S 128 1,575 / 1,548. So S K has to reach 3 (4 at 16 bits) times the
// texels. Small maps leave the fixed amount, more than a few probes' footprints
// from near caches: 300,000 points, R 2: K 4: S 32 262 / 431, S 128 695 / 809,
// K 8: S 64 682 / 615 (float32), 554 / 605 (16 bits), K 16, S 64 1,006 / 802;
// 1,000,000 points, float32, R 4, K 4, S 400: 5,313 / 6,922. Where the lanes
// are several a point, sharing its footprints' addresses costs them more:
// 100,000 points, float32, R 8, K 4, S 64: 262 / 232; S 128: 444 / 311; 60,000
// points, 16 bits, R 8, K 8, S 64: 203 / 190. (More than 128 directions have
// their footprints computed twice: 300,000 points, float32, R 4, K 4, S 400:
// 1,959 / 2,142, R 8: 2,087 / 1,937.)
// Calls of few points do not fill the machine with a thread a point: 21,907
// points, S 64: 276 / 220; 1,000: 204 / 170; and the fewer, the less a warp has
// to save (R 3, K 1, S 32: 16,384 points 72 / 83, 32,768: 83 / 103).
constexpr int64_t kPointSmall = 32768;
static bool shade_by_point(const QueryArgs& a)
{
    if (a.mode != SOP_MODE_SHADE || a.dir_world) return false;
    const int64_t t = point_texels(a.R), S = a.S, sk = S * a.K;
    if (sizeof(float4) * (size_t)S + kPointWarps * point_smem_bytes(a.R) > kSmemMost) return false;
    const bool f32 = a.rgbo_dtype == SOP_F32;
    if (a.M <= kPointSmall) {
        const int64_t least = f32 ? (a.M < 7500 ? a.M / 50 : 150) : a.M / 64;
        return sk >= t && sk >= least;
    }
    if (sk < (f32 ? 3 : 4) * t) return false;
    const int lanes = shade_lanes(a.rgbo_dtype, a.M);
    if (f32 && lanes >= 4) return sk >= 150;
    if (!f32 && lanes >= 8) return sk - S >= 400;
    if (f32 && lanes == 2) return sk - (S > 128 && t < 64 ? 4 : 2) * S >= 300;
    return sk - 3 * S >= 400 + t / 2;
}

template <int DT, int KMAX, int LANES>
static cudaError_t shadow_warp_launch(const ShadeK& k, cudaStream_t s)
{
    shadow_warp_kernel<DT, KMAX, LANES><<<(unsigned)((k.M + 255) / 256), 256, sizeof(float4) * (size_t)k.S, s>>>(k);
    return cudaGetLastError();
}
template <int DT, int KMAX>
static cudaError_t shadow_warp_dispatch(const ShadeK& k, cudaStream_t s)
{
    // (kShadowWarpPoints leaves one or two)
    if (DT == SOP_F32 && shade_lanes(DT, k.M) == 1) return shadow_warp_launch<DT, KMAX, 1>(k, s);
    return shadow_warp_launch<DT, KMAX, 2>(k, s);
}

template <int DT, int MODE>
static cudaError_t shade_k(const ShadeK& k, cudaStream_t s)
{
    if (MODE == SOP_MODE_SHADOW && k.S <= kShadowTab && k.M >= kShadowWarpPoints && k.K <= kShadowWarpK) {
        if (k.K <= 4) return shadow_warp_dispatch<DT, 4>(k, s);
        if (k.K <= 8) return shadow_warp_dispatch<DT, 8>(k, s);
        return shadow_warp_dispatch<DT, 16>(k, s);
    }
    if (k.K <= 4) return shade_dispatch<DT, 4, MODE>(k, s);
    if (k.K <= 8) return shade_dispatch<DT, 8, MODE>(k, s);
    if (k.K <= 16) return shade_dispatch<DT, 16, MODE>(k, s);
    return shade_dispatch<DT, 32, MODE>(k, s);
}

template <int DT, int KMAX, int MODE>
static cudaError_t shade_world_launch(const ShadeK& k, cudaStream_t s)
{
    const int bs = 256, LANES = shade_lanes(DT, k.M);
    const int64_t threads = k.M * LANES;
    const unsigned nb = (unsigned)((threads + bs - 1) / bs);
    const size_t smem = 3 * sizeof(float4) * (size_t)k.S;
    auto fn = shade_world_kernel<DT, KMAX, MODE>;
    if (const cudaError_t e = allow_smem(fn, smem); e != cudaSuccess) return e;
    fn<<<nb, bs, smem, s>>>(k, LANES);
    return cudaGetLastError();
}

template <int DT, int MODE>
static cudaError_t shade_world_k(const ShadeK& k, cudaStream_t s)
{
    if (k.K <= 4) return shade_world_launch<DT, 4, MODE>(k, s);
    if (k.K <= 8) return shade_world_launch<DT, 8, MODE>(k, s);
    if (k.K <= 16) return shade_world_launch<DT, 16, MODE>(k, s);
    return shade_world_launch<DT, 32, MODE>(k, s);
}

template <int DT>
static cudaError_t shade_mode(const ShadeK& k, int mode, bool world, cudaStream_t s)
{
    if (world)
        return mode == SOP_MODE_SHADE ? shade_world_k<DT, SOP_MODE_SHADE>(k, s) : shade_world_k<DT, SOP_MODE_SHADOW>(k, s);
    return mode == SOP_MODE_SHADE ? shade_k<DT, SOP_MODE_SHADE>(k, s) : shade_k<DT, SOP_MODE_SHADOW>(k, s);
}


cudaError_t launch_shade(const QueryArgs& a, const QueryLayout& L, char* ws, cudaStream_t s)
{
    if (a.M == 0) return cudaSuccess;
    ShadeK k;
    k.n = a.n;
    k.wo = a.wo;
    k.albedo = a.albedo;
    k.rough = a.rough;
    k.metal = a.metal;
    k.M = a.M;
    k.rgbo = a.rgbo;
    k.R = a.R;
    k.K = a.K;
    k.S = a.S;
    k.He = a.He;
    k.We = a.We;
    k.envq = reinterpret_cast<const float4*>(ws + L.envq);
    k.env_layout = a.env_layout;
    k.quads = ws + L.quads;
    k.dirs = reinterpret_cast<const float4*>(ws + L.dirs);
    k.idx = reinterpret_cast<const int32_t*>(ws + L.idx);
    k.w = reinterpret_cast<const float*>(ws + L.w);
    k.specular = a.specular;
    k.out = a.out;
    k.status = status_word();
    if (shade_by_point(a)) switch (a.rgbo_dtype) {
    case SOP_F32: return shade_point_k<SOP_F32>(k, s);
    case SOP_BF16: return shade_point_k<SOP_BF16>(k, s);
    case SOP_F16: return shade_point_k<SOP_F16>(k, s);
    default: return cudaErrorInvalidValue;
    }
    switch (a.rgbo_dtype) {
    case SOP_F32: return shade_mode<SOP_F32>(k, a.mode, a.dir_world != 0, s);
    case SOP_BF16: return shade_mode<SOP_BF16>(k, a.mode, a.dir_world != 0, s);
    case SOP_F16: return shade_mode<SOP_F16>(k, a.mode, a.dir_world != 0, s);
    default: return cudaErrorInvalidValue;
    }
}


// ---------------------------------------------------------------------------
// Multi-CTA build of the same quantised grid for large site sets (the
// single-CTA probe_grid_kernel is meant for thousands of probes).
// ---------------------------------------------------------------------------
__global__ void sites_bbox_kernel(const float* __restrict__ pos, int32_t N, int32_t* __restrict__ mm)
{
    int32_t lo[3] = {INT32_MAX, INT32_MAX, INT32_MAX}, hi[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        for (int a = 0; a < 3; ++a) {
            const int32_t q = quantise(pos[3 * i + a]);
            lo[a] = min(lo[a], q);
            hi[a] = max(hi[a], q);
        }
    cta_box_atomic(lo, hi, mm);
}

// one warp: the smallest cell edge of at most cap cells
__global__ void sites_setup_kernel(const int32_t* __restrict__ mm, int64_t cap, ProbeGrid* grid)
{
    uint32_t ext[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) ext[a] = (uint32_t)mm[3 + a] - (uint32_t)mm[a];
    const uint32_t cs = grid_edge(ext, cap, threadIdx.x);
    if (threadIdx.x != 0) return;
    ProbeGrid G;
    G.cs = (int32_t)cs;
    G.inv = 0xffffffffu / cs;
    G.ncells = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        G.qmin[a] = mm[a];
        G.dims[a] = (int32_t)(ext[a] / cs) + 1;
        G.ncells *= G.dims[a];
    }
    *grid = G;
}

__global__ void sites_zero_kernel(int32_t* __restrict__ cnt, int64_t n, int32_t* mm)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) cnt[i] = 0;
    if (i < 3) mm[i] = INT32_MAX;
    else if (i < 6) mm[i] = INT32_MIN;
}

__global__ void sites_count_kernel(const float* __restrict__ pos, int32_t N, const ProbeGrid* __restrict__ gp,
                                   int32_t* __restrict__ cnt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    atomicAdd(&cnt[grid_cell(*gp, quantise(pos[3 * i]), quantise(pos[3 * i + 1]), quantise(pos[3 * i + 2]))], 1);
}

__global__ void sites_fill_kernel(const float* __restrict__ pos, int32_t N, const ProbeGrid* __restrict__ gp,
                                  const int32_t* __restrict__ start, int32_t* __restrict__ cnt, int4* __restrict__ ent)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int32_t x = quantise(pos[3 * i]), y = quantise(pos[3 * i + 1]), z = quantise(pos[3 * i + 2]);
    const int cell = grid_cell(*gp, x, y, z);
    ent[start[cell] + atomicAdd(&cnt[cell], 1)] = make_int4(x, y, z, (int)i);
}

// ---------------------------------------------------------------------------
// K nearest sites (e.g. Gaussian centres) of M query points, exact, with the
// same integer keys and tie rule as the probe search.
// ---------------------------------------------------------------------------
size_t sites_grid_bytes(int32_t N)
{
    int g = 1;
    while ((int64_t)g * g * g < N) ++g;
    const int64_t cells = (int64_t)(g + 1) * (g + 1) * (g + 1);
    size_t o = align256(sizeof(ProbeGrid));
    o = align256(o + sizeof(int32_t) * (size_t)(cells + 1));
    o = align256(o + sizeof(int32_t) * (size_t)cells);
    o = align256(o + sizeof(int4) * (size_t)N);
    o = align256(o + 8 * sizeof(int32_t));
    o = align256(o + sizeof(long long) * scan_scratch_count(cells));
    return o;
}

// ---------------------------------------------------------------------------
// Read-bandwidth probe: every thread streams 16-byte loads over the buffer,
// `reps` times, on all SMs. A buffer that fits in L2 gives the L2-to-SM read
// rate that bounds the query's footprint gathers; a larger one the HBM rate.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512) read_probe_kernel(const uint4* __restrict__ buf, int64_t n16, int32_t reps,
                                                          float* __restrict__ sink)
{
    uint32_t acc = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int r = 0; r < reps; ++r)
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += stride) {
            const uint4 v = __ldcg(buf + i);
            acc ^= v.x ^ v.y ^ v.z ^ v.w;
        }
    // a store the compiler cannot drop, taken only for one improbable value
    if (acc == 0x9e3779b9u) sink[0] = (float)acc;
}

cudaError_t launch_read_probe(const void* buf, size_t bytes, int32_t reps, float* sink, cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    read_probe_kernel<<<(unsigned)(sms > 0 ? sms : 152) * 4, 512, 0, s>>>(reinterpret_cast<const uint4*>(buf),
                                                                             (int64_t)(bytes / 16), reps, sink);
    return cudaGetLastError();
}

SitesGrid launch_sites_grid(const float* sites, int32_t N, char* ws, cudaStream_t s)
{
    int g = 1;
    while ((int64_t)g * g * g < N) ++g;
    const int64_t cells = (int64_t)(g + 1) * (g + 1) * (g + 1);
    size_t o = 0;
    SitesGrid r;
    ProbeGrid* grid = reinterpret_cast<ProbeGrid*>(ws + o);
    o = align256(sizeof(ProbeGrid));
    int32_t* cstart = reinterpret_cast<int32_t*>(ws + o);
    o = align256(o + sizeof(int32_t) * (size_t)(cells + 1));
    int32_t* ccnt = reinterpret_cast<int32_t*>(ws + o);
    o = align256(o + sizeof(int32_t) * (size_t)cells);
    int4* ent = reinterpret_cast<int4*>(ws + o);
    o = align256(o + sizeof(int4) * (size_t)N);
    int32_t* mm = reinterpret_cast<int32_t*>(ws + o);
    o = align256(o + 8 * sizeof(int32_t));
    long long* scan = reinterpret_cast<long long*>(ws + o);
    if (N <= 16384) {
        probe_grid_kernel<<<1, 1024, 0, s>>>(sites, N, g, grid, cstart, ccnt, ent);
    } else {
        const unsigned nb = (unsigned)((N + 255) / 256);
        sites_zero_kernel<<<(unsigned)((cells + 255) / 256), 256, 0, s>>>(ccnt, cells, mm);
        sites_bbox_kernel<<<nb < kBoxCtas ? nb : kBoxCtas, 256, 0, s>>>(sites, N, mm);
        // about 4 sites per grid cell: the warp search pays per ring (a
        // round of dependent loads) far more than per candidate (32 lanes)
        const int64_t cap = N / 4 > 4096 ? N / 4 : 4096;
        sites_setup_kernel<<<1, 32, 0, s>>>(mm, cap < cells ? cap : cells, grid);
        sites_count_kernel<<<nb, 256, 0, s>>>(sites, N, grid, ccnt);
        ScanArgs sa;
        sa.n = &grid->ncells;
        sa.cnt = ccnt;
        sa.start = cstart;
        sa.scratch = scan;
        launch_scan(sa, cap < cells ? cap : cells, ScanNoFinal{}, s);
        sites_fill_kernel<<<nb, 256, 0, s>>>(sites, N, grid, cstart, ccnt, ent);
    }
    r.grid = grid;
    r.cell_start = cstart;
    r.entries = ent;
    return r;
}


// ===========================================================================
// Allocation-free variant of the query + shade (sop_query_shade_noalloc).
//
// For callers that cannot allocate device memory themselves. Its scratch is
// one file-scope device array of kNoAllocScratchBytes, present on every GPU
// that loads the library until the process exits. Host code cannot pass the
// array's name to a kernel (on the host it is only a stand-in symbol), so the
// first call on each device looks up the array's device address with
// cudaGetSymbolAddress while that device is current, and later calls reuse
// it. The probe atlas and the environment are read in the caller's own
// layouts (no repacked copies), and points are processed in chunks of
// kNoAllocChunk so that the per-point neighbour lists fit the array. All
// calls share the array: calls that overlap on the GPU (other streams, other
// host threads) race on it.
// ===========================================================================
constexpr size_t kNoAllocScratchBytes = size_t(8) << 20;
constexpr int64_t kNoAllocChunk = 16384;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

size_t noalloc_scratch_bytes() { return kNoAllocScratchBytes; }
int64_t noalloc_chunk() { return kNoAllocChunk; }

// Bilinear environment lookup straight from the caller's [He][We][3] array.
__device__ __forceinline__ float3 env_lookup_direct(const float* __restrict__ env, int He, int We, float3 w)
{
    const float th = atan2f(sqrtf(w.x * w.x + w.y * w.y), w.z);
    const float ph = atan2f(w.y, w.x);
    const float s = (ph + kPi) * kInv2Pi * We - 0.5f;
    const float t = th * kInvPi * He - 0.5f;
    const float fs = floorf(s), ft = floorf(t);
    const float a = s - fs, b = t - ft;
    int c0 = (int)fs;
    c0 = c0 < 0 ? c0 + We : c0;
    c0 = min(max(c0, 0), We - 1);
    const int c1 = c0 + 1 == We ? 0 : c0 + 1;
    const int r0 = min(max((int)ft, 0), He - 1), r1 = min(max((int)ft + 1, 0), He - 1);
    const float* e00 = env + ((int64_t)r0 * We + c0) * 3;
    const float* e01 = env + ((int64_t)r0 * We + c1) * 3;
    const float* e10 = env + ((int64_t)r1 * We + c0) * 3;
    const float* e11 = env + ((int64_t)r1 * We + c1) * 3;
    const float w00 = (1.f - a) * (1.f - b), w01 = a * (1.f - b), w10 = (1.f - a) * b, w11 = a * b;
    return f3(w00 * __ldg(e00) + w01 * __ldg(e01) + w10 * __ldg(e10) + w11 * __ldg(e11),
              w00 * __ldg(e00 + 1) + w01 * __ldg(e01 + 1) + w10 * __ldg(e10 + 1) + w11 * __ldg(e11 + 1),
              w00 * __ldg(e00 + 2) + w01 * __ldg(e01 + 2) + w10 * __ldg(e10 + 2) + w11 * __ldg(e11 + 2));
}

// Equirectangular -> octahedral environment (Sec. 4.1): texel (i, j) of the
// [H][H] map takes the bilinear equirectangular value at its centre
// direction (computed in double, rounded once).
__global__ void env_to_oct_kernel(const float* __restrict__ env, int32_t He, int32_t We, float* __restrict__ out,
                                  int32_t H)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (int64_t)H * H) return;
    double d[3];
    oct_decode_centre_f64(H, (int)(k % H), (int)(k / H), d);
    const float3 v = env_lookup_direct(env, He, We, f3((float)d[0], (float)d[1], (float)d[2]));
    out[3 * k] = v.x;
    out[3 * k + 1] = v.y;
    out[3 * k + 2] = v.z;
}

cudaError_t launch_env_to_oct(const float* env, int32_t He, int32_t We, float* out, int32_t H, cudaStream_t s)
{
    const int64_t n = (int64_t)H * H;
    env_to_oct_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(env, He, We, out, H);
    return cudaGetLastError();
}

struct ShadeDirectK {
    const float *n, *wo, *albedo, *rough, *metal;
    int64_t M;
    const void* rgbo;
    int32_t R, K, S, He, We;
    const float* env;
    const float4* dirs;
    const int32_t* idx;
    const float* w;
    float specular;
    float* out;
};

// One thread per point; texels read from the gutter atlas, four per probe.
template <int DT, int KMAX, int MODE>
__global__ void __launch_bounds__(256) shade_direct_kernel(const ShadeDirectK a)
{
    using TX = Texel<DT>;
    extern __shared__ float4 s_dirs[];
    for (int i = threadIdx.x; i < a.S; i += blockDim.x) s_dirs[i] = a.dirs[i];
    __syncthreads();
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= a.M) return;
    const float3 nr = load3(a.n, m);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 n = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    float3 tt, bb;
    onb(n, tt, bb);
    const float3 wo = load3(a.wo, m);
    const int RS = a.R + 2;
    const typename TX::raw* atlas = reinterpret_cast<const typename TX::raw*>(a.rgbo);
    int64_t base[KMAX];
    float W[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const bool on = k < a.K;
        base[k] = on ? (int64_t)__ldg(a.idx + m * a.K + k) * RS * RS : 0;
        W[k] = on ? __ldg(a.w + m * a.K + k) : 0.f;
    }
    float3 kd = f3(0.f, 0.f, 0.f), F0 = f3(0.f, 0.f, 0.f);
    float a2 = 0.f, kk = 0.f, specV = 0.f;
    if (MODE == SOP_MODE_SHADE) {
        const float3 alb = load3(a.albedo, m);
        const float r = __ldg(a.rough + m), mt = __ldg(a.metal + m);
        const float dsc = (1.f - mt) * kInvPi;
        kd = f3(dsc * alb.x, dsc * alb.y, dsc * alb.z);
        const float f0d = 0.08f * a.specular * (1.f - mt);
        F0 = f3(f0d + alb.x * mt, f0d + alb.y * mt, f0d + alb.z * mt);
        const float al = r * r;
        a2 = al * al;
        kk = (r + 1.f) * (r + 1.f) * 0.125f;
        const float NdotV = fmaxf(dot3(n, wo), 1e-4f);
        specV = (NdotV / (NdotV * (1.f - kk) + kk)) / (4.f * NdotV);
    }
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, den0 = 0.f, den1 = 0.f, den2 = 0.f;
    const float Rf = (float)a.R;
    for (int i = 0; i < a.S; ++i) {
        const float4 l = s_dirs[i];
        const float3 w = f3(fmaf(l.x, tt.x, fmaf(l.y, bb.x, l.z * n.x)), fmaf(l.x, tt.y, fmaf(l.y, bb.y, l.z * n.y)),
                            fmaf(l.x, tt.z, fmaf(l.y, bb.z, l.z * n.z)));
        const float2 uv = oct_encode(w);
        const float s = uv.x * Rf - 0.5f, t = uv.y * Rf - 0.5f;
        const float fi = floorf(s), fj = floorf(t);
        const float fu = s - fi, fv = t - fj;
        const int i0 = min(max((int)fi + 1, 0), a.R), j0 = min(max((int)fj + 1, 0), a.R);
        const int off = j0 * RS + i0;
        const float w00 = (1.f - fu) * (1.f - fv), w10 = fu * (1.f - fv), w01 = (1.f - fu) * fv, w11 = fu * fv;
        float4 pr = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            if (k < a.K) {
                const typename TX::raw* p = atlas + base[k] + off;
                const float4 t00 = TX::load(p), t10 = TX::load(p + 1), t01 = TX::load(p + RS), t11 = TX::load(p + RS + 1);
                const float c00 = W[k] * w00, c10 = W[k] * w10, c01 = W[k] * w01, c11 = W[k] * w11;
                pr.x += c00 * t00.x + c10 * t10.x + c01 * t01.x + c11 * t11.x;
                pr.y += c00 * t00.y + c10 * t10.y + c01 * t01.y + c11 * t11.y;
                pr.z += c00 * t00.z + c10 * t10.z + c01 * t01.z + c11 * t11.z;
                pr.w += c00 * t00.w + c10 * t10.w + c01 * t01.w + c11 * t11.w;
            }
        }
        const float3 Ld = env_lookup_direct(a.env, a.He, a.We, w);
        const float NdotL = l.z;
        const float vis = 1.f - pr.w;
        if (MODE == SOP_MODE_SHADE) {
            float3 h = w + wo;
            const float hl2 = dot3(h, h);
            h = hl2 > 1e-30f ? rsqrtf(hl2) * h : n;
            const float NdotH = dot3(n, h), VdotH = dot3(wo, h);
            const float3 cr = cross3(n, h);
            const float sin2 = dot3(cr, cr);
            const float den = NdotH * NdotH * a2 + sin2;
            const float D = __fdividef(a2, kPi * den * den);
            const float spec = __fdividef(D * specV, NdotL * (1.f - kk) + kk);
            const float x1 = 1.f - VdotH, x2 = x1 * x1, fc = x2 * x2 * x1;
            acc0 += (kd.x + spec * (F0.x + (1.f - F0.x) * fc)) * (vis * Ld.x + pr.x) * NdotL;
            acc1 += (kd.y + spec * (F0.y + (1.f - F0.y) * fc)) * (vis * Ld.y + pr.y) * NdotL;
            acc2 += (kd.z + spec * (F0.z + (1.f - F0.z) * fc)) * (vis * Ld.z + pr.z) * NdotL;
        } else {
            acc0 += Ld.x * vis * NdotL;
            acc1 += Ld.y * vis * NdotL;
            acc2 += Ld.z * vis * NdotL;
            den0 += Ld.x * NdotL;
            den1 += Ld.y * NdotL;
            den2 += Ld.z * NdotL;
        }
    }
    float* o = a.out + 3 * m;
    if (MODE == SOP_MODE_SHADE) {
        const float sc = 2.f * kPi / (float)a.S;
        o[0] = sc * acc0;
        o[1] = sc * acc1;
        o[2] = sc * acc2;
    } else {
        o[0] = den0 < 1e-20f ? 1.f : acc0 / den0;
        o[1] = den1 < 1e-20f ? 1.f : acc1 / den1;
        o[2] = den2 < 1e-20f ? 1.f : acc2 / den2;
    }
}

template <int DT, int KMAX, int MODE>
static cudaError_t shade_direct_launch(const ShadeDirectK& k, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * (size_t)k.S;
    auto fn = shade_direct_kernel<DT, KMAX, MODE>;
    if (const cudaError_t e = allow_smem(fn, smem); e != cudaSuccess) return e;
    fn<<<(unsigned)((k.M + 255) / 256), 256, smem, s>>>(k);
    return cudaGetLastError();
}

template <int DT, int MODE>
static cudaError_t shade_direct_k(const ShadeDirectK& k, cudaStream_t s)
{
    if (k.K <= 4) return shade_direct_launch<DT, 4, MODE>(k, s);
    if (k.K <= 8) return shade_direct_launch<DT, 8, MODE>(k, s);
    if (k.K <= 16) return shade_direct_launch<DT, 16, MODE>(k, s);
    return shade_direct_launch<DT, 32, MODE>(k, s);
}

template <int DT>
static cudaError_t shade_direct_mode(const ShadeDirectK& k, int mode, cudaStream_t s)
{
    return mode == SOP_MODE_SHADE ? shade_direct_k<DT, SOP_MODE_SHADE>(k, s) : shade_direct_k<DT, SOP_MODE_SHADOW>(k, s);
}

// Device address of the scratch array on the current device, looked up once
// per device (the lookup must run with that device current).
static cudaError_t noalloc_scratch_ptr(char** out)
{
    static std::mutex mu;
    static char* ptrs[256] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!ptrs[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        ptrs[dev] = static_cast<char*>(p);
    }
    *out = ptrs[dev];
    return cudaSuccess;
}

// Scratch layout for P probes, S directions and K neighbours (per chunk).
static QueryLayout noalloc_layout(int32_t P, int32_t K, int32_t S)
{
    QueryLayout L{};
    int g = 1;
    while ((int64_t)g * g * g < P) ++g;
    L.g_axis = g;
    L.cells_cap = (g + 1) * (g + 1) * (g + 1);
    size_t o = 0;
    L.grid_hdr = o;   o = align256(o + sizeof(ProbeGrid));
    L.cell_start = o; o = align256(o + sizeof(int32_t) * (size_t)(L.cells_cap + 1));
    L.cell_cnt = o;   o = align256(o + sizeof(int32_t) * (size_t)L.cells_cap);
    L.entries = o;    o = align256(o + sizeof(int4) * (size_t)P);
    L.dirs = o;       o = align256(o + sizeof(float4) * (size_t)S);
    L.idx = o;        o = align256(o + sizeof(int32_t) * (size_t)kNoAllocChunk * K);
    L.w = o;          o = align256(o + sizeof(float) * (size_t)kNoAllocChunk * K);
    L.total = o;
    return L;
}

size_t noalloc_required_bytes(int32_t P, int32_t K, int32_t S) { return noalloc_layout(P, K, S).total; }

cudaError_t launch_query_noalloc(const QueryArgs& a, cudaStream_t s)
{
    char* ws = nullptr;
    cudaError_t e = noalloc_scratch_ptr(&ws);
    if (e != cudaSuccess) return e;
    const QueryLayout L = noalloc_layout(a.P, a.K, a.S);
    if (L.total > kNoAllocScratchBytes) return cudaErrorInvalidValue;  // checked by the caller first
    ProbeGrid* grid = reinterpret_cast<ProbeGrid*>(ws + L.grid_hdr);
    int32_t* cstart = reinterpret_cast<int32_t*>(ws + L.cell_start);
    int32_t* ccnt = reinterpret_cast<int32_t*>(ws + L.cell_cnt);
    int4* ent = reinterpret_cast<int4*>(ws + L.entries);
    float4* dirs = reinterpret_cast<float4*>(ws + L.dirs);
    int32_t* idx = reinterpret_cast<int32_t*>(ws + L.idx);
    float* w = reinterpret_cast<float*>(ws + L.w);
    // the grid build clears its own counters, so stale contents are harmless
    probe_grid_kernel<<<1, 1024, 0, s>>>(a.probe_pos, a.P, L.g_axis, grid, cstart, ccnt, ent);
    dirs_kernel<<<(a.S + 127) / 128, 128, 0, s>>>(a.S, a.dirs_local, dirs, nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int64_t m0 = 0; m0 < a.M; m0 += kNoAllocChunk) {
        const int64_t mc = a.M - m0 < kNoAllocChunk ? a.M - m0 : kNoAllocChunk;
        KnnK kn;
        kn.x = a.x + 3 * m0;
        kn.nrm = a.n + 3 * m0;
        kn.M = mc;
        kn.K = a.K;
        kn.P = a.P;
        kn.snap_key = a.snap_key;
        kn.r2_key = a.r2_key;
        kn.grid = grid;
        kn.cell_start = cstart;
        kn.entries = ent;
        kn.probe_pos = a.probe_pos;
        kn.ws_idx = idx;
        kn.ws_w = w;
        kn.user_idx = a.out_idx ? a.out_idx + m0 * a.K : nullptr;
        kn.user_w = a.out_w ? a.out_w + m0 * a.K : nullptr;
        kn.status = status_word();
        if ((e = launch_knn(kn, s)) != cudaSuccess) return e;
        ShadeDirectK k;
        k.n = a.n + 3 * m0;
        k.wo = a.wo + 3 * m0;
        k.albedo = a.albedo + 3 * m0;
        k.rough = a.rough + m0;
        k.metal = a.metal + m0;
        k.M = mc;
        k.rgbo = a.rgbo;
        k.R = a.R;
        k.K = a.K;
        k.S = a.S;
        k.He = a.He;
        k.We = a.We;
        k.env = a.env;
        k.dirs = dirs;
        k.idx = idx;
        k.w = w;
        k.specular = a.specular;
        k.out = a.out + 3 * m0;
        switch (a.rgbo_dtype) {
        case SOP_F32: e = shade_direct_mode<SOP_F32>(k, a.mode, s); break;
        case SOP_BF16: e = shade_direct_mode<SOP_BF16>(k, a.mode, s); break;
        case SOP_F16: e = shade_direct_mode<SOP_F16>(k, a.mode, s); break;
        default: e = cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace sop
