// Importance-sampled light directions for rendering (Sec. 4.2, Eq. PDF:
// density H W I / (4 pi) over the texels of the octahedral environment).
//   imp_max_kernel     intensity I_t = r + g + b of every texel (float32, in
//                      this order), each CTA's maximum;
//   imp_q_kernel       q_t = max(1, floor(I_t / I_max 2^20)), one tile of
//                      texels a CTA, and the tile's sum;
//   imp_sample_kernel  one warp a sample: sample i takes the texel t whose
//                      interval [C_{t-1}, C_t) of the running sums of q holds
//                      floor((2i + 1) Q / (2S)) (exact integers; the tile
//                      from the tile sums, the texel within it), its centre
//                      direction (double, rounded once) and density
//                      H^2 q_t / (4 pi Q).
// All three are short passes over the texels (4 bytes of q each in between);
// the running sums themselves are never stored. For a 512 x 512 environment
// and 64 samples they take 4 + 8 + 16 us (each launch timed alone); with the
// running sums formed by one CTA, whose 1,024 threads walked a contiguous
// chunk each, twice, with a double division per texel, 1,619 us.
#include <math.h>

#include "sop_device.cuh"
#include "sop_internal.h"

namespace sop {

constexpr int kImpThreads = 256;
constexpr int kImpTile = 2048;     // texels of one tile (8 a thread)
constexpr int kImpMaxTiles = 2048; // H <= 2048
constexpr int kImpMaxCtas = 512;   // of imp_max_kernel

struct ImpK {
    const float* env;
    int64_t T;        // texels
    int32_t H, S, n_max, n_tiles;
    int64_t* tile;    // [n_tiles] sums of q
    uint32_t* cmax;   // [n_max] largest intensity a CTA, as float bits
    int32_t* q;       // [T]
    float4* out;
};

__device__ __forceinline__ float imp_intensity(const float* __restrict__ env, int64_t t)
{
    return env[3 * t] + env[3 * t + 1] + env[3 * t + 2];
}

// intensities are >= 0 here, so their order is that of their bits
__global__ void __launch_bounds__(kImpThreads) imp_max_kernel(const ImpK k)
{
    __shared__ uint32_t s_max;
    if (threadIdx.x == 0) s_max = 0u;
    __syncthreads();
    uint32_t best = 0u;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < k.T; t += (int64_t)gridDim.x * blockDim.x)
        best = max(best, __float_as_uint(fmaxf(imp_intensity(k.env, t), 0.f)));
    best = __reduce_max_sync(0xffffffffu, best);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, best);
    __syncthreads();
    if (threadIdx.x == 0) k.cmax[blockIdx.x] = s_max;
}

// A non-negative float as mant 2^exp, mant an integer below 2^24.
__device__ __forceinline__ uint32_t float_mant(float v, int& e)
{
    const uint32_t b = __float_as_uint(v), x = b >> 23;
    e = x ? (int)x : 1;
    return (b & 0x7fffffu) | (x ? 0x800000u : 0u);
}

// max(1, floor(I / imax 2^20)), exactly: a float quotient is within one of
// the floor, and integer products decide. (The quotient rounded to double
// has the same floor: an exact quotient below an integer N <= 2^20 lies at
// least 1 / mant(imax) > 2^-24 below it, far more than a double's rounding.)
// Anything but 0 < I, 0 < imax < inf gives 1.
__device__ __forceinline__ int32_t imp_q(float I, float imax)
{
    if (!(I > 0.f) || !(imax > 0.f) || !isfinite(imax)) return 1;
    int ei, em;
    const uint32_t a = float_mant(I, ei), b = float_mant(imax, em);
    const int sh = 20 + ei - em;  // I <= imax, so a 2^sh < 2^45
    if (sh < 0) return 1;
    const uint64_t num = (uint64_t)a << sh;
    int64_t q = (int64_t)(I / imax * 1048576.f);
    if ((uint64_t)q * b > num) --q;
    else if ((uint64_t)(q + 1) * b <= num) ++q;
    return q < 1 ? 1 : (int32_t)q;
}

__global__ void __launch_bounds__(kImpThreads) imp_q_kernel(const ImpK k)
{
    __shared__ uint32_t s_max, s_sum;  // (2048 texels of at most 2^20: the sum fits)
    if (threadIdx.x == 0) {
        s_max = 0u;
        s_sum = 0u;
    }
    __syncthreads();
    uint32_t best = 0u;
    for (int i = threadIdx.x; i < k.n_max; i += kImpThreads) best = max(best, k.cmax[i]);
    best = __reduce_max_sync(0xffffffffu, best);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, best);
    __syncthreads();
    const float imax = __uint_as_float(s_max);
    uint32_t sum = 0u;
#pragma unroll
    for (int j = 0; j < kImpTile / kImpThreads; ++j) {
        const int64_t t = (int64_t)blockIdx.x * kImpTile + j * kImpThreads + threadIdx.x;
        if (t >= k.T) break;
        const int32_t q = imp_q(imp_intensity(k.env, t), imax);
        k.q[t] = q;
        sum += (uint32_t)q;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, sum);
    __syncthreads();
    if (threadIdx.x == 0) k.tile[blockIdx.x] = (int64_t)s_sum;
}

__global__ void __launch_bounds__(kImpThreads) imp_sample_kernel(const ImpK k)
{
    constexpr int NW = kImpThreads / 32, PER = kImpMaxTiles / kImpThreads, RND = kImpTile / 128;
    __shared__ int64_t s_cum[kImpMaxTiles];  // inclusive sums of the tiles
    __shared__ int64_t s_w[NW];
    __shared__ int64_t s_at[NW];  // the warps' texels and their q
    __shared__ int32_t s_q[NW];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t v[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int t = threadIdx.x * PER + j;
        sum += t < k.n_tiles ? k.tile[t] : 0;
        v[j] = sum;
    }
    int64_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(full, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    int64_t base = inc - sum;
    for (int w = 0; w < warp; ++w) base += s_w[w];
#pragma unroll
    for (int j = 0; j < PER; ++j) s_cum[threadIdx.x * PER + j] = base + v[j];
    __syncthreads();
    const int i = min((int)(blockIdx.x * NW) + warp, k.S - 1);
    const int64_t Q = s_cum[k.n_tiles - 1];
    const int64_t target = (2 * (int64_t)i + 1) * Q / (2 * (int64_t)k.S);
    int lo = 0, hi = k.n_tiles - 1;  // smallest tile whose inclusive sum exceeds the target
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (s_cum[mid] > target) hi = mid;
        else lo = mid + 1;
    }
    // within the tile, what is left of the target fits 32 bits
    uint32_t left = (uint32_t)(target - (lo > 0 ? s_cum[lo - 1] : 0));
    const int64_t t0 = (int64_t)lo * kImpTile + 4 * lane;
    int64_t at = 0;
    int32_t q = 1;
    for (int r = 0; r < RND; ++r) {
        const int64_t t = t0 + 128 * r;
        int4 c = make_int4(0, 0, 0, 0);
        if (t + 3 < k.T) c = *reinterpret_cast<const int4*>(k.q + t);
        else if (t < k.T) c = make_int4(k.q[t], t + 1 < k.T ? k.q[t + 1] : 0, t + 2 < k.T ? k.q[t + 2] : 0, 0);
        const uint32_t mine = (uint32_t)c.x + (uint32_t)c.y + (uint32_t)c.z + (uint32_t)c.w;
        const uint32_t all = __reduce_add_sync(full, mine);
        if (left >= all) {
            left -= all;
            continue;
        }
        uint32_t upto = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(full, upto, o);
            if (lane >= o) upto += u;
        }
        const int win = __ffs(__ballot_sync(full, upto > left)) - 1;
        uint32_t rest = left - (upto - mine);  // (of the winning lane)
        int j = 0;
        q = c.x;
        if (rest >= (uint32_t)q) { rest -= q; j = 1; q = c.y; }
        if (j == 1 && rest >= (uint32_t)q) { rest -= q; j = 2; q = c.z; }
        if (j == 2 && rest >= (uint32_t)q) { j = 3; q = c.w; }
        at = __shfl_sync(full, t + j, win);
        q = __shfl_sync(full, q, win);
        break;
    }
    // the direction and density in double, a lane a sample of the CTA's
    if (lane == 0) {
        s_at[warp] = at;
        s_q[warp] = q;
    }
    __syncthreads();
    const int o = blockIdx.x * NW + lane;
    if (warp != 0 || lane >= NW || o >= k.S) return;
    at = s_at[lane];
    double d[3];
    oct_decode_centre_f64(k.H, (int)(at % k.H), (int)(at / k.H), d);
    const double pdf = (double)k.T * (double)s_q[lane] / (4.0 * 3.14159265358979323846 * (double)Q);
    k.out[o] = make_float4((float)d[0], (float)d[1], (float)d[2], (float)pdf);
}

size_t importance_ws_bytes(int32_t H)
{
    return align256(sizeof(unsigned int)) + align256(sizeof(int64_t) * (size_t)H * H);
}

cudaError_t launch_importance_dirs(const float* env, int32_t H, int32_t S, float* out, char* ws, cudaStream_t s)
{
    ImpK k;
    k.env = env;
    k.H = H;
    k.S = S;
    k.T = (int64_t)H * H;
    k.n_tiles = (int32_t)((k.T + kImpTile - 1) / kImpTile);
    const int64_t nb = (k.T + 4 * kImpThreads - 1) / (4 * kImpThreads);
    k.n_max = (int32_t)(nb < kImpMaxCtas ? nb : kImpMaxCtas);
    // tile sums, CTA maxima and q, packed (less than importance_ws_bytes for every H)
    k.tile = reinterpret_cast<int64_t*>(ws);
    k.cmax = reinterpret_cast<uint32_t*>(ws + 8 * (size_t)k.n_tiles);
    k.q = reinterpret_cast<int32_t*>(ws + ((8 * (size_t)k.n_tiles + 4 * (size_t)k.n_max + 15) & ~(size_t)15));
    k.out = reinterpret_cast<float4*>(out);
    imp_max_kernel<<<(unsigned)k.n_max, kImpThreads, 0, s>>>(k);
    imp_q_kernel<<<(unsigned)k.n_tiles, kImpThreads, 0, s>>>(k);
    imp_sample_kernel<<<(unsigned)((S + kImpThreads / 32 - 1) / (kImpThreads / 32)), kImpThreads, 0, s>>>(k);
    return cudaGetLastError();
}

}  // namespace sop
