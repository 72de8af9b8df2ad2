// One warp per shading point: the blended probe map of the point.
//
// The footprint of a light direction lies at the same place of every probe's
// octahedral map (the maps are in the world frame), so the K-probe blend of
// Eq. 5 can be taken before the bilinear fetch instead of after it: the warp
// blends the map texels that its S directions touch once, into shared
// memory, and every direction then reads four texels there instead of 4 K
// from the atlas. About half of the (R + 2)^2 stored texels lie above a
// point's horizon, and they are read in rows, 16 or 8 bytes a lane next to
// one another, so K fetches a texel cost less than 4 K gathers a direction as
// soon as the directions outnumber half of the texels.
#pragma once
#include "sop_device.cuh"

namespace sop {

constexpr int kPointWarps = 8;  // warps (points) a CTA

// Shared memory of one warp: the blended map, the marks and list of the
// texels in use.
struct PointSmem {
    float4* map;      // [(R+2)^2] (RGB, O), by stored texel
    uint32_t* mark;   // [words]
    uint16_t* list;   // [(R+2)^2]
};
__host__ __device__ inline int point_texels(int R) { return (R + 2) * (R + 2); }
__host__ __device__ inline int point_words(int R) { return (point_texels(R) + 31) / 32; }
__host__ __device__ inline size_t point_smem_bytes(int R)
{
    const size_t t = (size_t)point_texels(R);
    return ((16 * t + 4 * (size_t)(point_words(R) + 1) + 2 * t) + 15) & ~(size_t)15;
}
__device__ __forceinline__ PointSmem point_smem(char* base, int R)
{
    const int t = point_texels(R);
    PointSmem s;
    s.map = reinterpret_cast<float4*>(base);
    s.mark = reinterpret_cast<uint32_t*>(base + 16 * (size_t)t);
    s.list = reinterpret_cast<uint16_t*>(base + 16 * (size_t)t + 4 * (size_t)(point_words(R) + 1));
    return s;
}

// Footprint of a direction: base stored texel and the fractions in it.
struct Foot {
    int off;
    float fu, fv;
};
__device__ __forceinline__ Foot oct_foot(float3 w, float Rf, int R)
{
    const float2 uv = oct_encode(w);
    const float s = uv.x * Rf - 0.5f, t = uv.y * Rf - 0.5f;
    const float fi = floorf(s), fj = floorf(t);
    Foot f;
    f.fu = s - fi;
    f.fv = t - fj;
    const int i0 = min(max((int)fi + 1, 0), R), j0 = min(max((int)fj + 1, 0), R);
    f.off = j0 * (R + 2) + i0;
    return f;
}

// marks the four texels of a footprint
__device__ __forceinline__ void point_mark(const PointSmem& s, int off, int RS)
{
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int o = off + r * RS, w = o >> 5;
        const uint64_t bits = (uint64_t)3u << (o & 31);
        atomicOr(s.mark + w, (uint32_t)bits);
        if (bits >> 32) atomicOr(s.mark + w + 1, 1u);
    }
}

// the marked texels, in order, into the list; returns their number
__device__ __forceinline__ int point_list(const PointSmem& s, int words, int lane)
{
    int n = 0;
    for (int w = 0; w < words; ++w) {
        const uint32_t m = s.mark[w];
        if ((m >> lane) & 1u) s.list[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(w * 32 + lane);
        n += __popc(m);
    }
    return n;
}

}  // namespace sop
