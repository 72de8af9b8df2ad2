// Automatic placement of SOPs (Sec. 3.2) for sm_103a: farthest point
// sampling (FPS) of a surface point cloud, then an offset of the chosen
// points along their normals.
//
// Distances are exact integer squared distances of positions quantised to
// 2^-20 (the query's keys), so every choice is exact and matches a plain
// sequential FPS: the first point is `start`, each next one has the largest
// smallest key to the chosen ones, ties to the lower index.
//
// The k choices are a serial chain, so the time is the number of its links
// times the time of one. Both are cut:
//  - Several choices a link. The points are sorted into spatially compact
//    pieces (a Morton-ordered counting sort), one piece a CTA. Each CTA
//    publishes its best point and the exact best that would be left in its
//    piece after that one; a leader takes the published points in order of
//    key for as long as the sequential order is certain: the next one's key
//    must not be lowered by a point taken in this link, and no piece already
//    drawn from may hold a larger (or equal) key. On an object's surface
//    that is about 10 of 4,096 choices a link.
//  - Work only where something changes. Positions and keys stay in registers
//    (5 words a point), a warp's points are compact, and a warp whose box
//    lies beyond its largest key from a chosen point skips the update.
// One link is then two exchanges through L2 (the pieces' bests to the leader,
// the choices back), each a set of 16-byte words that carry their round's
// tag, polled until the tag is there: no counters, no fences. The launch is
// cooperative (the CTAs wait on one another); waits are bounded.
//
// 750,710 points, 4,096 choices: 73.1 ms with one choice a link in one
// 16-CTA cluster whose slices lay in L2; 26.6 ms with the points in the
// registers of all SMs and one choice a link, every CTA polling every other
// (the polls crowd L2); 1.69 to 1.79 ms as described (395 links of about 9,000
// cycles: a third the leader's ranking, a third the two exchanges). On a
// lattice, where ties leave one choice a link, 10,648 points and 4,096 choices
// take 12.0 ms (22.0 in the cluster).
#include <climits>

#include "scan.cuh"
#include "sop_device.cuh"
#include "sop_internal.h"

namespace sop {

constexpr int kFpsThreads = 512;
constexpr int kFpsWarps = kFpsThreads / 32;
constexpr int kFpsMaxCtas = 160;
constexpr int kFpsPicks = 32;   // choices a link at most (one a lane)
constexpr int kFpsCopies = 8;   // of the list of choices, to spread its readers
constexpr int kFpsRegPoints = 512;  // points of a warp that stay in registers (16 a thread)
// Up to this many points one CTA takes them all (0.9 us a choice; 0.3 us in
// all CTAs from 4,096 points): fewer do not leave room for the exchange in
// the workspace, which is sized by the points.
constexpr int64_t kFpsOneCta = 2048;
// polls of one exchange before it gives up (an L2 round trip each: seconds)
constexpr int kFpsPollMax = 1 << 22;

// One CTA's answer in a link; every word carries the link's tag.
struct FpsSlot {
    ulonglong2 a;  // key of its best point; index | tag << 32
    ulonglong2 b;  // x | y << 32; z | tag << 32
    ulonglong2 c;  // largest key left without that point; far flag | tag << 32
    ulonglong2 pad;
};

struct FpsK {
    const float* pts;
    const float* nrm;
    int64_t n, chunk, start;  // chunk: points of a CTA
    int32_t k, per_warp;      // per_warp: points of a warp
    float offset;
    const int32_t* perm;      // points in Morton order, or NULL: their own order
    FpsSlot* slots;           // [2][gridDim.x], cleared before the launch
    ulonglong2* list;         // [2][kFpsCopies][kFpsPicks]: x, y, z, tag * 2 + used; cleared too
    unsigned long long* gd;   // keys, when the points do not fit in registers
    int64_t* out_idx;
    float* out_pos;
    unsigned int* status;
};

__device__ __forceinline__ int3 quant3(const float* p, int64_t i)
{
    // x 2^20 is exact in float; rintf rounds half to even
    return make_int3((int)rintf(__ldg(p + 3 * i) * 1048576.f), (int)rintf(__ldg(p + 3 * i + 1) * 1048576.f),
                     (int)rintf(__ldg(p + 3 * i + 2) * 1048576.f));
}

// ---- Morton-ordered counting sort ---------------------------------------------
// mm: [0, 3) smallest and [3, 6) largest quantised coordinates, [6] cells
__global__ void fps_clear_kernel(int32_t* __restrict__ cnt, int32_t cells, int32_t* __restrict__ mm)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < cells) cnt[i] = 0;
    if (i < 3) mm[i] = INT_MAX;
    else if (i < 6) mm[i] = INT_MIN;
    else if (i == 6) mm[i] = cells;
}

__global__ void fps_bbox_kernel(const float* __restrict__ pts, int64_t n, int32_t* __restrict__ mm)
{
    int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int3 q = quant3(pts, i);
        lo[0] = min(lo[0], q.x); lo[1] = min(lo[1], q.y); lo[2] = min(lo[2], q.z);
        hi[0] = max(hi[0], q.x); hi[1] = max(hi[1], q.y); hi[2] = max(hi[2], q.z);
    }
    cta_box_atomic(lo, hi, mm);
}

// Cubic cells, 2^bits an axis over the longest side of the points' box, in
// Morton order. (Only the order of the points depends on it, no result.)
__device__ __forceinline__ uint32_t fps_cell(const int32_t* __restrict__ mm, int bits, int3 q)
{
    uint32_t ext = 0;
    for (int a = 0; a < 3; ++a) ext = max(ext, (uint32_t)mm[3 + a] - (uint32_t)mm[a]);
    const int sh = max(0, 32 - __clz(ext) - bits);
    uint32_t m = 0;
    const uint32_t c[3] = {((uint32_t)q.x - (uint32_t)mm[0]) >> sh, ((uint32_t)q.y - (uint32_t)mm[1]) >> sh,
                           ((uint32_t)q.z - (uint32_t)mm[2]) >> sh};
    for (int b = 0; b < bits; ++b)
        for (int a = 0; a < 3; ++a) m |= ((c[a] >> b) & 1u) << (3 * b + a);
    return m;
}

__global__ void fps_count_kernel(const float* __restrict__ pts, int64_t n, const int32_t* __restrict__ mm, int bits,
                                 int32_t* __restrict__ cnt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) atomicAdd(&cnt[fps_cell(mm, bits, quant3(pts, i))], 1);
}

__global__ void fps_fill_kernel(const float* __restrict__ pts, int64_t n, const int32_t* __restrict__ mm, int bits,
                                const int32_t* __restrict__ start, int32_t* __restrict__ cnt, int32_t* __restrict__ perm)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t c = fps_cell(mm, bits, quant3(pts, i));
    perm[start[c] + atomicAdd(&cnt[c], 1)] = (int32_t)i;
}

// ---- the links ------------------------------------------------------------------
// 16-byte words of an exchange, each read and written as one access
__device__ __forceinline__ void word_store(ulonglong2* p, unsigned long long lo, unsigned long long hi)
{
    asm volatile("{\n .reg .b128 v;\n mov.b128 v, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], v;\n}" ::"l"(p), "l"(lo),
                 "l"(hi)
                 : "memory");
}
__device__ __forceinline__ ulonglong2 word_load(const ulonglong2* p)
{
    ulonglong2 r;
    asm volatile("{\n .reg .b128 v;\n ld.relaxed.gpu.global.b128 v, [%2];\n mov.b128 {%0, %1}, v;\n}"
                 : "=l"(r.x), "=l"(r.y)
                 : "l"(p)
                 : "memory");
    return r;
}
__device__ __forceinline__ unsigned long long pack2(uint32_t lo, uint32_t hi)
{
    return (unsigned long long)lo | (unsigned long long)hi << 32;
}

__device__ __forceinline__ unsigned long long fps_key(int3 a, int3 b)
{
    // |a - b| as unsigned: right for any pair of int32
    const uint32_t dx = (uint32_t)max(a.x, b.x) - (uint32_t)min(a.x, b.x),
                   dy = (uint32_t)max(a.y, b.y) - (uint32_t)min(a.y, b.y),
                   dz = (uint32_t)max(a.z, b.z) - (uint32_t)min(a.z, b.z);
    return (unsigned long long)dx * dx + (unsigned long long)dy * dy + (unsigned long long)dz * dz;
}
// Points within [-2^30, 2^30) (positions below 1024): differences fit in
// int32 and no sum of squares wraps. Links with any other point take one
// choice each and skip no update.
__device__ __forceinline__ bool fps_near(int3 a)
{
    const int m = 1 << 30;
    return a.x >= -m && a.x < m && a.y >= -m && a.y < m && a.z >= -m && a.z < m;
}
__device__ __forceinline__ unsigned long long fps_key_near(int3 a, int3 b)
{
    const int dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    return (unsigned long long)((long long)dx * dx) + (unsigned long long)((long long)dy * dy) +
           (unsigned long long)((long long)dz * dz);
}
// smallest squared distance of p to the box [lo, hi] (near points)
__device__ __forceinline__ unsigned long long fps_box(int3 lo, int3 hi, int3 p)
{
    const int dx = max(max(lo.x - p.x, p.x - hi.x), 0), dy = max(max(lo.y - p.y, p.y - hi.y), 0),
              dz = max(max(lo.z - p.z, p.z - hi.z), 0);
    return (unsigned long long)((long long)dx * dx) + (unsigned long long)((long long)dy * dy) +
           (unsigned long long)((long long)dz * dz);
}

__device__ __forceinline__ unsigned long long warp_max(unsigned long long key)
{
    const uint32_t hi = (uint32_t)(key >> 32);
    const uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? (uint32_t)key : 0u);
    return pack2(ml, mh);
}
// Lane that holds the warp's best: the largest key, ties to the lowest index.
__device__ __forceinline__ int warp_best(unsigned long long key, uint32_t idx)
{
    const bool top = key == warp_max(key);
    const uint32_t mi = __reduce_min_sync(0xffffffffu, top ? idx : 0xffffffffu);
    return __ffs(__ballot_sync(0xffffffffu, top && idx == mi)) - 1;
}

// PT: points a thread keeps in registers; 0: positions are read again and
// the keys kept in the workspace.
template <int PT>
__global__ void __launch_bounds__(kFpsThreads, 1) fps_kernel(const FpsK k)
{
    __shared__ uint32_t s_id[PT > 0 ? PT * kFpsThreads : 1];
    __shared__ unsigned long long s_key[kFpsWarps], s_left[kFpsWarps];  // a warp's best; what a choice would leave
    __shared__ uint32_t s_idx[kFpsWarps];
    __shared__ int3 s_pos[kFpsWarps];
    // leader: the candidates among the CTAs' answers, and the best of each of its warps
    __shared__ unsigned long long s_ckey[kFpsMaxCtas], s_tkey[kFpsMaxCtas / 32], s_tleft[kFpsMaxCtas / 32], s_bad;
    __shared__ uint32_t s_cidx[kFpsMaxCtas], s_tidx[kFpsMaxCtas / 32];
    __shared__ int3 s_cpos[kFpsMaxCtas];
    __shared__ int s_rank[kFpsMaxCtas], s_m;
    __shared__ int3 s_pick[kFpsPicks];
    __shared__ int s_np, s_lost, s_far;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ctas = (int)gridDim.x;
    const bool leader = blockIdx.x == 0;
    const int64_t c0 = (int64_t)blockIdx.x * k.chunk, c1 = min(k.n, c0 + k.chunk);
    const int64_t lo = min(c1, c0 + (int64_t)warp * k.per_warp), hi = min(c1, lo + k.per_warp);
    int3 q[PT > 0 ? PT : 1];
    unsigned long long d[PT > 0 ? PT : 1];
    int3 bl = make_int3(INT_MAX, INT_MAX, INT_MAX), bh = make_int3(INT_MIN, INT_MIN, INT_MIN);
    bool near = true;
    const auto extend = [&](int3 v) {
        bl = make_int3(min(bl.x, v.x), min(bl.y, v.y), min(bl.z, v.z));
        bh = make_int3(max(bh.x, v.x), max(bh.y, v.y), max(bh.z, v.z));
        near = near && fps_near(v);
    };
    if (PT > 0) {
#pragma unroll
        for (int j = 0; j < PT; ++j) {
            const int64_t i = lo + j * 32 + lane;
            const bool in = i < hi;
            const int32_t id = in ? (k.perm ? k.perm[i] : (int32_t)i) : -1;
            s_id[j * kFpsThreads + threadIdx.x] = (uint32_t)id;
            q[j] = in ? quant3(k.pts, id) : make_int3(0, 0, 0);
            d[j] = in ? ULLONG_MAX : 0ull;  // a slot past the end never wins
            if (in) extend(q[j]);
        }
    } else {
        for (int64_t i = lo + lane; i < hi; i += 32) {
            extend(quant3(k.pts, k.perm[i]));
            k.gd[i] = ULLONG_MAX;
        }
    }
    bl = make_int3(__reduce_min_sync(full, bl.x), __reduce_min_sync(full, bl.y), __reduce_min_sync(full, bl.z));
    bh = make_int3(__reduce_max_sync(full, bh.x), __reduce_max_sync(full, bh.y), __reduce_max_sync(full, bh.z));
    if (threadIdx.x == 0) {
        s_lost = s_far = 0;
        s_np = 1;
        s_pick[0] = quant3(k.pts, k.start);
        if (leader) k.out_idx[0] = k.start;
    }
    unsigned long long wmax = lo < hi ? ULLONG_MAX : 0ull;  // largest key of the warp's points
    near = __syncthreads_and(near);
    int done = 0;
    for (uint32_t tag = 1;; ++tag) {
        // ---- the choices of the last link: new keys, and the warp's best
        const int np = s_np;
        // lane p tests choice p against the warp's box
        const int3 mp = lane < np ? s_pick[lane] : make_int3(0, 0, 0);
        const bool mex = near && fps_near(mp);
        unsigned hit = __ballot_sync(full, lane < np && !(mex && fps_box(bl, bh, mp) >= wmax));
        const bool dirty = hit != 0u || tag == 1;
        for (; hit; hit &= hit - 1) {
            const int p = __ffs(hit) - 1;
            const int3 c = s_pick[p];
            const bool exact = near && fps_near(c);
            if (PT > 0) {
                if (exact) {
#pragma unroll
                    for (int j = 0; j < PT; ++j) {
                        const unsigned long long key = fps_key_near(q[j], c);
                        d[j] = key < d[j] ? key : d[j];
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < PT; ++j) {
                        const unsigned long long key = fps_key(q[j], c);
                        d[j] = key < d[j] ? key : d[j];
                    }
                }
            } else {
                for (int64_t i = lo + lane; i < hi; i += 32) {
                    const unsigned long long key = fps_key(quant3(k.pts, k.perm[i]), c);
                    if (key < k.gd[i]) k.gd[i] = key;
                }
            }
        }
        done += np;
        if (done >= k.k) break;
        if (dirty) {
            unsigned long long m = 0ull;
            uint32_t id = 0xffffffffu;
            int3 at = make_int3(0, 0, 0);
            if (PT > 0) {
#pragma unroll
                for (int j = 0; j < PT; ++j) m = d[j] > m ? d[j] : m;
            } else {
                for (int64_t i = lo + lane; i < hi; i += 32) m = k.gd[i] > m ? k.gd[i] : m;
            }
            wmax = warp_max(m);
            if (m == wmax) {  // few lanes: the lowest index among the points that have it
                if (PT > 0) {
#pragma unroll
                    for (int j = 0; j < PT; ++j)
                        if (d[j] == wmax) {
                            const uint32_t v = s_id[j * kFpsThreads + threadIdx.x];
                            if (v < id) {
                                id = v;
                                at = q[j];
                            }
                        }
                } else {
                    for (int64_t i = lo + lane; i < hi; i += 32)
                        if (k.gd[i] == wmax && (uint32_t)k.perm[i] < id) id = (uint32_t)k.perm[i];
                    if (id != 0xffffffffu) at = quant3(k.pts, id);
                }
            }
            __syncwarp();
            const uint32_t best = __reduce_min_sync(full, id);
            if (id == best && (id != 0xffffffffu || lane == 0)) {
                s_key[warp] = wmax;
                s_idx[warp] = id;
                s_pos[warp] = at;
            }
        }
        __syncthreads();
        // ---- the CTA's best, and the largest key that it would leave
        const bool on = lane < kFpsWarps;
        const unsigned long long wk = on ? s_key[lane] : 0ull;
        const uint32_t wi = on ? s_idx[lane] : 0xffffffffu;
        const int wb = warp_best(wk, wi);
        const int3 bp = s_pos[wb];
        unsigned long long left = wmax;
        if (ctas > 1 && near && fps_box(bl, bh, bp) < wmax) {
            left = 0ull;
            if (PT > 0) {
#pragma unroll
                for (int j = 0; j < PT; ++j) {
                    const unsigned long long key = fps_key_near(q[j], bp), v = key < d[j] ? key : d[j];
                    left = v > left ? v : left;
                }
            } else {
                for (int64_t i = lo + lane; i < hi; i += 32) {
                    const unsigned long long key = fps_key_near(quant3(k.pts, k.perm[i]), bp), e = k.gd[i],
                                             v = key < e ? key : e;
                    left = v > left ? v : left;
                }
            }
            left = warp_max(left);
        }
        if (lane == 0) s_left[warp] = left;
        __syncthreads();
        if (ctas == 1) {
            if (warp == 0 && lane == wb) {
                s_pick[0] = bp;
                s_np = 1;
                k.out_idx[done] = wi;
            }
            __syncthreads();
            continue;
        }
        // ---- to the leader. A slot is written again two links later: the
        // leader has read it before it published the choices of its link
        FpsSlot* sl = k.slots + (size_t)(tag & 1u) * ctas;
        ulonglong2* list = k.list + (size_t)(tag & 1u) * kFpsCopies * kFpsPicks;
        if (warp == 0) {
            const unsigned long long cl = warp_max(on ? s_left[lane] : 0ull);
            if (lane == wb) {
                word_store(&sl[blockIdx.x].a, wk, pack2(wi, tag));
                word_store(&sl[blockIdx.x].b, pack2((uint32_t)bp.x, (uint32_t)bp.y), pack2((uint32_t)bp.z, tag));
                word_store(&sl[blockIdx.x].c, cl, pack2(near ? 0u : 1u, tag));
            }
            __syncwarp();
        }
        if (leader) {
            unsigned long long mk = 0ull;
            uint32_t mi = 0xffffffffu;
            int3 mc = make_int3(0, 0, 0);
            if (threadIdx.x < kFpsMaxCtas) {
                const int c = (int)threadIdx.x;
                ulonglong2 a = make_ulonglong2(0ull, 0ull), b = a, e = a;
                bool have = c >= ctas;
                for (int tries = 0; !__all_sync(full, have) && tries < kFpsPollMax; ++tries) {
                    if (!have) {
                        a = word_load(&sl[c].a);
                        b = word_load(&sl[c].b);
                        e = word_load(&sl[c].c);
                        have = (uint32_t)(a.y >> 32) == tag && (uint32_t)(b.y >> 32) == tag && (uint32_t)(e.y >> 32) == tag;
                    }
                }
                if (!have) s_lost = 1;
                if ((uint32_t)e.y) s_far = 1;
                mk = c < ctas ? a.x : 0ull;
                mi = c < ctas ? (uint32_t)a.y : 0xffffffffu;
                mc = make_int3((int)(uint32_t)b.x, (int)(uint32_t)(b.x >> 32), (int)(uint32_t)b.y);
                const int w = warp_best(mk, mi);
                const unsigned long long l = warp_max(e.x);
                if (lane == w) {
                    s_tkey[warp] = mk;
                    s_tidx[warp] = mi;
                    s_tleft[warp] = l;
                }
            }
            if (threadIdx.x == 0) {
                s_m = s_np = 0;
                s_bad = 0ull;
            }
            __syncthreads();
            // candidates: the best of all, and those above every key that a
            // choice could leave unseen
            if (threadIdx.x < kFpsMaxCtas) {
                unsigned long long tk = s_tkey[0], tl = s_tleft[0];
                uint32_t ti = s_tidx[0];
#pragma unroll
                for (int w = 1; w < kFpsMaxCtas / 32; ++w) {
                    const unsigned long long v = s_tkey[w], l = s_tleft[w];
                    const uint32_t vi = s_tidx[w];
                    const bool up = v > tk || (v == tk && vi < ti);
                    tk = up ? v : tk;
                    ti = up ? vi : ti;
                    tl = l > tl ? l : tl;
                }
                if ((int)threadIdx.x < ctas && (mk > tl || (mk == tk && mi == ti))) {
                    const int j = atomicAdd(&s_m, 1);
                    s_ckey[j] = mk;
                    s_cidx[j] = mi;
                    s_cpos[j] = mc;
                    s_rank[j] = 0;
                }
            }
            __syncthreads();
            // each candidate's rank, and the largest key that a candidate
            // ranked above would lower: the order is certain above it
            const int m = s_m;
            for (int i0 = 0; i0 < m; i0 += 32) {
                const int i = i0 + lane;
                const unsigned long long ki = i < m ? s_ckey[i] : 0ull;
                const uint32_t ii = i < m ? s_cidx[i] : 0xffffffffu;
                const int3 pi = i < m ? s_cpos[i] : make_int3(0, 0, 0);
                int above = 0;
                bool bad = false;
                for (int j = warp; j < m; j += kFpsWarps) {
                    const unsigned long long kj = s_ckey[j];
                    const bool up = kj > ki || (kj == ki && s_cidx[j] < ii);
                    above += up ? 1 : 0;
                    bad = bad || (up && fps_key(s_cpos[j], pi) < ki);
                }
                if (i < m && above) atomicAdd(&s_rank[i], above);
                if (i < m && bad) atomicMax(&s_bad, ki);
            }
            __syncthreads();
            const int most = s_far ? 1 : min(kFpsPicks, k.k - done);
            for (int i = threadIdx.x; i < m; i += kFpsThreads) {
                const int r = s_rank[i];
                if (r < most && (r == 0 || s_ckey[i] > s_bad)) {
                    s_pick[r] = s_cpos[i];
                    k.out_idx[done + r] = s_cidx[i];
                    atomicAdd(&s_np, 1);
                }
            }
            __syncthreads();
            if (warp < kFpsCopies && !s_lost) {
                const int3 p = lane < s_np ? s_pick[lane] : make_int3(0, 0, 0);
                word_store(list + warp * kFpsPicks + lane, pack2((uint32_t)p.x, (uint32_t)p.y),
                           pack2((uint32_t)p.z, tag * 2u + (lane < s_np ? 1u : 0u)));
            }
        } else if (warp == 0) {
            const ulonglong2* e = list + (blockIdx.x % kFpsCopies) * kFpsPicks + lane;
            ulonglong2 v = make_ulonglong2(0ull, 0ull);
            bool have = false;
            for (int tries = 0; !__all_sync(full, have) && tries < kFpsPollMax; ++tries) {
                if (!have) {
                    v = word_load(e);
                    have = (uint32_t)(v.y >> 33) == tag;
                }
            }
            if (!have) s_lost = 1;
            const bool used = ((v.y >> 32) & 1ull) != 0ull;
            if (used) s_pick[lane] = make_int3((int)(uint32_t)v.x, (int)(uint32_t)(v.x >> 32), (int)(uint32_t)v.y);
            const int cnt = __popc(__ballot_sync(full, used));
            if (lane == 0) s_np = cnt;
        }
        __syncthreads();
        if (s_lost) {  // a CTA did not answer
            if (threadIdx.x == 0 && k.status) atomicOr(k.status, SOP_DEVSTAT_TIMEOUT);
            return;
        }
    }
    if (!leader || !k.out_pos) return;
    __syncthreads();  // out_idx, written by this CTA
    for (int it = threadIdx.x; it < k.k; it += kFpsThreads) {
        const int64_t i = k.out_idx[it];
        for (int a = 0; a < 3; ++a) {
            const double x = k.pts[3 * i + a];
            k.out_pos[3 * it + a] = (float)(k.nrm ? x + (double)k.offset * (double)k.nrm[3 * i + a] : x);
        }
    }
}

size_t fps_ws_bytes(int64_t n) { return align256(16 * (size_t)n) + align256(8 * (size_t)n); }

// Morton cells: about a quarter to one a point (a surface fills a small part
// of its box), 4 to 128 an axis
static int fps_cell_bits(int64_t n)
{
    int b = 2;
    while (b < 7 && ((int64_t)1 << (3 * (b + 1))) <= n) ++b;
    return b;
}

template <int PT>
static cudaError_t fps_launch(FpsK a, int ctas, cudaStream_t s)
{
    void* args[] = {&a};
    return cudaLaunchCooperativeKernel(reinterpret_cast<void*>(fps_kernel<PT>), dim3(ctas), dim3(kFpsThreads), args, 0, s);
}

cudaError_t launch_fps(const float* pts, const float* nrm, int64_t n, int32_t k, int64_t start, float offset,
                       int64_t* out_idx, float* out_pos, char* ws, cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int ctas = n <= kFpsOneCta || sms < 1 ? 1 : (sms > kFpsMaxCtas ? kFpsMaxCtas : sms);
    FpsK a;
    a.pts = pts;
    a.nrm = nrm;
    a.n = n;
    a.chunk = (n + ctas - 1) / ctas;
    a.per_warp = (int32_t)((a.chunk + kFpsWarps - 1) / kFpsWarps);
    a.start = start;
    a.k = k;
    a.offset = offset;
    a.out_idx = out_idx;
    a.out_pos = out_pos;
    a.status = status_word();
    a.perm = nullptr;
    a.slots = nullptr;
    a.list = nullptr;
    a.gd = nullptr;
    if (n > kFpsOneCta) {
        // workspace: the order, the exchange (cleared here: a word of an
        // earlier call would carry a valid tag), the sort's cells, and the
        // keys where they do not stay in registers
        const int bits = fps_cell_bits(n);
        const int32_t cells = 1 << (3 * bits);
        size_t o = 0;
        int32_t* perm = reinterpret_cast<int32_t*>(ws);
        o = align256(4 * (size_t)n);
        a.slots = reinterpret_cast<FpsSlot*>(ws + o);
        a.list = reinterpret_cast<ulonglong2*>(a.slots + 2 * (size_t)ctas);
        const size_t exch = 2 * sizeof(FpsSlot) * (size_t)ctas + 2 * sizeof(ulonglong2) * kFpsCopies * kFpsPicks;
        o = align256(o + exch);
        int32_t* mm = reinterpret_cast<int32_t*>(ws + o);
        o = align256(o + 8 * sizeof(int32_t));
        int32_t* cnt = reinterpret_cast<int32_t*>(ws + o);
        o = align256(o + 4 * (size_t)cells);
        ScanArgs sa;
        sa.n = mm + 6;
        sa.cnt = cnt;
        sa.start = reinterpret_cast<int32_t*>(ws + o);
        o = align256(o + 4 * (size_t)(cells + 1));
        sa.scratch = reinterpret_cast<long long*>(ws + o);
        o = align256(o + sizeof(long long) * scan_scratch_count(cells));
        if (a.per_warp > kFpsRegPoints) {
            a.gd = reinterpret_cast<unsigned long long*>(ws + o);
            o += 8 * (size_t)n;
        }
        // (holds for every n > kFpsOneCta: cells <= n, at most 160 CTAs)
        if (o > fps_ws_bytes(n)) return cudaErrorInvalidValue;
        if ((e = cudaMemsetAsync(a.slots, 0, exch, s)) != cudaSuccess) return e;
        const unsigned nb = (unsigned)((n + 255) / 256), nz = (unsigned)((cells + 255) / 256);
        fps_clear_kernel<<<nz, 256, 0, s>>>(cnt, cells, mm);
        fps_bbox_kernel<<<nb < kBoxCtas ? nb : kBoxCtas, 256, 0, s>>>(pts, n, mm);
        fps_count_kernel<<<nb, 256, 0, s>>>(pts, n, mm, bits, cnt);
        launch_scan(sa, cells, ScanNoFinal{}, s);
        fps_fill_kernel<<<nb, 256, 0, s>>>(pts, n, mm, bits, sa.start, cnt, perm);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        a.perm = perm;
    }
    // Points a thread: one, or the next even number. A slot past the end costs
    // what a point costs, two of them 5 to 6% of the call (4,096 choices, us:
    // 400,000 points in 6 / 8 slots 1,459 / 1,541; 700,000 in 10 / 12 / 16
    // 1,759 / 1,875 / 2,074; 850,000 in 12 / 16 1,864 / 2,063; 1,000,000 in 14 /
    // 16 2,023 / 2,111).
    switch (a.per_warp <= 32 ? 1 : 2 * ((a.per_warp + 63) / 64)) {
    case 1: return fps_launch<1>(a, ctas, s);
    case 2: return fps_launch<2>(a, ctas, s);
    case 4: return fps_launch<4>(a, ctas, s);
    case 6: return fps_launch<6>(a, ctas, s);
    case 8: return fps_launch<8>(a, ctas, s);
    case 10: return fps_launch<10>(a, ctas, s);
    case 12: return fps_launch<12>(a, ctas, s);
    case 14: return fps_launch<14>(a, ctas, s);
    case 16: return fps_launch<16>(a, ctas, s);
    default: return fps_launch<0>(a, ctas, s);  // (more than kFpsRegPoints a warp)
    }
}

}  // namespace sop
