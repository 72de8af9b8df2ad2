// Hand-written adjoint of the SOP query/shade (SHADE mode) for sm_103a.
//
// The environment map, the materials and the SOP textures are the learnable
// quantities of the paper's decomposition step (Sec. 3.1.2, Eq. 3-6; the SOP
// textures are optimised under trace guidance). Given dL/dC [M,3] this kernel
// returns dL/d{albedo, roughness, metallic, raw normal} per point and
// accumulates dL/d{environment texels, probe texels}. Nothing of the forward
// pass is stored: every per-direction term is recomputed (frame, octahedral
// coordinates, K bilinear fetches, environment, BRDF), then pushed back
// through the same chain. Probe-texel gradients of border texels are folded
// back onto the texel the border copies, so the gradient is w.r.t. the
// compact [P][R][R] maps. Environment and probe gradients are scattered with
// float atomics (order-nondeterministic sums).
//
// Two kernels (adjoint_by_tile says which): adjoint_tile_kernel, eight points
// a CTA with a gradient image each in shared memory, and adjoint_kernel, a
// thread a point with K 4 vector atomics a direction into the maps. Both take
// the points grouped by their nearest probe (a counting sort), so that a
// CTA's points share probes, and accumulate the environment gradient as
// float4 texels (4 vector atomics a direction instead of 12 scalar ones),
// folded into g_env after.
#include "point_blend.cuh"
#include "sop_device.cuh"
#include "sop_internal.h"

namespace sop {

struct AdjK {
    const float *x, *n, *wo, *albedo, *rough, *metal;
    int64_t M;
    const void* rgbo;
    int32_t R, K, S, He, We;
    const float* env;
    const float4* dirs;
    const int32_t* idx;
    const float* w;
    const float* probe_pos;
    float specular;
    const float* grad_out;
    unsigned int* status;  // device status word or NULL
    float *g_albedo, *g_rough, *g_metal, *g_normal, *g_env;
    float4* g_maps;  // [P][R][R] (d rgb, d O)
    const int32_t* perm;  // order in which the points are taken
    float4* genv4;        // [He][We] environment gradient (rgb, -)
};

template <int DT, int KMAX>
__global__ void __launch_bounds__(128) adjoint_kernel(const AdjK a)
{
    using TX = Texel<DT>;
    extern __shared__ float4 s_dirs[];
    for (int i = threadIdx.x; i < a.S; i += blockDim.x) s_dirs[i] = a.dirs[i];
    __syncthreads();
    const int64_t pos = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // position in the grouped order
    if (pos >= a.M) return;
    const int64_t m = __ldg(a.perm + pos);

    const float3 nr = load3(a.n, m);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 n = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    float3 tt, bb;
    onb(n, tt, bb);
    const float3 wo = load3(a.wo, m);
    const float3 alb = load3(a.albedo, m);
    const float r = __ldg(a.rough + m), mt = __ldg(a.metal + m);
    const float3 go = load3(a.grad_out, m);
    if (a.status && !isfinite(go.x + go.y + go.z + alb.x + alb.y + alb.z + r + mt + wo.x + wo.y + wo.z))
        atomicOr(a.status, SOP_DEVSTAT_NONFINITE);
    const int RS = a.R + 2;
    const typename TX::raw* atlas = reinterpret_cast<const typename TX::raw*>(a.rgbo);
    int32_t pid[KMAX];
    float W[KMAX], gW[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const bool on = k < a.K;
        pid[k] = on ? __ldg(a.idx + m * a.K + k) : 0;
        W[k] = on ? __ldg(a.w + m * a.K + k) : 0.f;
        gW[k] = 0.f;
    }

    // per-point BRDF constants
    const float al = r * r, a2 = al * al, kk = (r + 1.f) * (r + 1.f) * 0.125f;
    const float NdotVraw = dot3(n, wo);
    const bool vclamp = NdotVraw < 1e-4f;
    const float NdotV = vclamp ? 1e-4f : NdotVraw;
    const float gvv = NdotV * (1.f - kk) + kk;
    const float G1V = NdotV / gvv;
    const float dG1V_dk = -NdotV * (1.f - NdotV) / (gvv * gvv);
    const float f0d = 0.08f * a.specular * (1.f - mt);
    const float F0[3] = {f0d + alb.x * mt, f0d + alb.y * mt, f0d + alb.z * mt};
    const float av[3] = {alb.x, alb.y, alb.z};
    const float gov[3] = {go.x, go.y, go.z};
    const float sc = 2.f * kPi / (float)a.S;
    // frame derivatives (Duff et al. 2017): dt/dn and db/dn, row = component
    const float sg = n.z >= 0.f ? 1.f : -1.f, aa = -1.f / (sg + n.z), a2n = aa * aa;
    const float dt[3][3] = {{2.f * sg * n.x * aa, 0.f, sg * n.x * n.x * a2n},
                            {sg * n.y * aa, sg * n.x * aa, sg * n.x * n.y * a2n},
                            {-sg, 0.f, 0.f}};
    const float db[3][3] = {{n.y * aa, n.x * aa, n.x * n.y * a2n}, {0.f, 2.f * n.y * aa, n.y * n.y * a2n},
                            {0.f, -1.f, 0.f}};
    float ga[3] = {0.f, 0.f, 0.f}, gr = 0.f, gm = 0.f, gn[3] = {0.f, 0.f, 0.f};
    const float Rf = (float)a.R;

    // neighbouring points (nearly the same frame) start their direction loops
    // S/32 apart, by their index, so that the lanes of a warp scatter into
    // other texels at each step instead of all into the same ones; the start
    // depends on the point alone, so each point's sums keep one order from
    // call to call whatever lane it lands in
    const int i_first = (int)(((m & 31) * (int64_t)a.S) >> 5);
    for (int ii = 0; ii < a.S; ++ii) {
        const int i = ii + i_first < a.S ? ii + i_first : ii + i_first - a.S;
        const float4 l = s_dirs[i];
        const float3 w = f3(fmaf(l.x, tt.x, fmaf(l.y, bb.x, l.z * n.x)), fmaf(l.x, tt.y, fmaf(l.y, bb.y, l.z * n.y)),
                            fmaf(l.x, tt.z, fmaf(l.y, bb.z, l.z * n.z)));
        const float NdotL = l.z;
        // ---- probe terms and their uv-derivatives ----------------------------
        const float2 uv = oct_encode(w);
        const float s = uv.x * Rf - 0.5f, t = uv.y * Rf - 0.5f;
        const float fi = floorf(s), fj = floorf(t);
        const float fu = s - fi, fv = t - fj;
        const int i0 = min(max((int)fi + 1, 0), a.R), j0 = min(max((int)fj + 1, 0), a.R);
        const int off = j0 * RS + i0;
        const float w00 = (1.f - fu) * (1.f - fv), w10 = fu * (1.f - fv), w01 = (1.f - fu) * fv, w11 = fu * fv;
        float4 pr = make_float4(0.f, 0.f, 0.f, 0.f), ps = pr, pt = pr;  // value, d/ds, d/dt
        float4 tk[KMAX];  // per-probe bilinear values (for dL/dW)
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            tk[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < a.K) {
                const typename TX::raw* p = atlas + (int64_t)pid[k] * RS * RS + off;
                const float4 t00 = TX::load(p), t10 = TX::load(p + 1), t01 = TX::load(p + RS),
                             t11 = TX::load(p + RS + 1);
                const float4 v = make_float4(w00 * t00.x + w10 * t10.x + w01 * t01.x + w11 * t11.x,
                                             w00 * t00.y + w10 * t10.y + w01 * t01.y + w11 * t11.y,
                                             w00 * t00.z + w10 * t10.z + w01 * t01.z + w11 * t11.z,
                                             w00 * t00.w + w10 * t10.w + w01 * t01.w + w11 * t11.w);
                tk[k] = v;
                const float Wk = W[k];
                pr.x += Wk * v.x; pr.y += Wk * v.y; pr.z += Wk * v.z; pr.w += Wk * v.w;
                // d/ds = (1-fv)(t10-t00) + fv(t11-t01); d/dt = (1-fu)(t01-t00) + fu(t11-t10)
                ps.x += Wk * ((1.f - fv) * (t10.x - t00.x) + fv * (t11.x - t01.x));
                ps.y += Wk * ((1.f - fv) * (t10.y - t00.y) + fv * (t11.y - t01.y));
                ps.z += Wk * ((1.f - fv) * (t10.z - t00.z) + fv * (t11.z - t01.z));
                ps.w += Wk * ((1.f - fv) * (t10.w - t00.w) + fv * (t11.w - t01.w));
                pt.x += Wk * ((1.f - fu) * (t01.x - t00.x) + fu * (t11.x - t10.x));
                pt.y += Wk * ((1.f - fu) * (t01.y - t00.y) + fu * (t11.y - t10.y));
                pt.z += Wk * ((1.f - fu) * (t01.z - t00.z) + fu * (t11.z - t10.z));
                pt.w += Wk * ((1.f - fu) * (t01.w - t00.w) + fu * (t11.w - t10.w));
            }
        }
        const float O = pr.w;
        const float Lin[3] = {pr.x, pr.y, pr.z};
        // ---- environment and its direction derivative ------------------------
        const float rho2 = w.x * w.x + w.y * w.y, rho = sqrtf(rho2);
        const float th = atan2f(rho, w.z), ph = atan2f(w.y, w.x);
        const float es = (ph + kPi) * kInv2Pi * a.We - 0.5f, et = th * kInvPi * a.He - 0.5f;
        const float fes = floorf(es), fet = floorf(et);
        const float ea = es - fes, eb = et - fet;
        int c0 = (int)fes;
        c0 = c0 < 0 ? c0 + a.We : c0;
        c0 = min(max(c0, 0), a.We - 1);
        const int c1 = c0 + 1 == a.We ? 0 : c0 + 1;
        const int r0 = min(max((int)fet, 0), a.He - 1), r1 = min(max((int)fet + 1, 0), a.He - 1);
        const int64_t ei[4] = {((int64_t)r0 * a.We + c0) * 3, ((int64_t)r0 * a.We + c1) * 3,
                               ((int64_t)r1 * a.We + c0) * 3, ((int64_t)r1 * a.We + c1) * 3};
        const float ew[4] = {(1.f - ea) * (1.f - eb), ea * (1.f - eb), (1.f - ea) * eb, ea * eb};
        float Ld[3], dLs[3], dLt[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float e00 = __ldg(a.env + ei[0] + c), e01 = __ldg(a.env + ei[1] + c), e10 = __ldg(a.env + ei[2] + c),
                        e11 = __ldg(a.env + ei[3] + c);
            Ld[c] = ew[0] * e00 + ew[1] * e01 + ew[2] * e10 + ew[3] * e11;
            dLs[c] = (1.f - eb) * (e01 - e00) + eb * (e11 - e10);
            dLt[c] = (1.f - ea) * (e10 - e00) + ea * (e11 - e01);
        }
        // ds/dw, dt/dw
        float dsw[3] = {0.f, 0.f, 0.f}, dtw[3] = {0.f, 0.f, 0.f};
        if (rho2 > 0.f) {
            const float ks = a.We * kInv2Pi / rho2;
            dsw[0] = -ks * w.y;
            dsw[1] = ks * w.x;
            const float r2 = rho2 + w.z * w.z, kt = a.He * kInvPi / r2;
            dtw[0] = kt * w.z * w.x / rho;
            dtw[1] = kt * w.z * w.y / rho;
            dtw[2] = -kt * rho;
        }
        // ---- BRDF ---------------------------------------------------------------
        const float3 hv = w + wo;
        const float hl = sqrtf(dot3(hv, hv));
        const float3 h = hl > 1e-30f ? (1.f / hl) * hv : n;
        const float NdotH = dot3(n, h), VdotH = dot3(wo, h);
        const float3 cr = cross3(n, h);
        const float sin2 = dot3(cr, cr);
        const float den = NdotH * NdotH * a2 + sin2;
        const float D = a2 / (kPi * den * den);
        const float gl = NdotL * (1.f - kk) + kk;
        const float G1L = NdotL / gl;
        const float spec_t = D * G1L * G1V / (4.f * NdotL * NdotV);
        const float x1 = 1.f - VdotH, x2 = x1 * x1, fc = x2 * x2 * x1;
        const float dD_da2 = (den - 2.f * a2 * NdotH * NdotH) / (kPi * den * den * den);
        const float dG1L_dk = -NdotL * (1.f - NdotL) / (gl * gl);
        const float dspec_dr =
            (dD_da2 * 4.f * r * r * r * G1L * G1V + D * (dG1L_dk * G1V + G1L * dG1V_dk) * (r + 1.f) * 0.25f) /
            (4.f * NdotL * NdotV);
        const float Gc = G1L * G1V / (4.f * NdotL * NdotV);
        const float dD_dNH = -4.f * a2 * a2 * NdotH / (kPi * den * den * den);
        const float dD_ds2 = -2.f * a2 / (kPi * den * den * den);
        float GN = 0.f, GS = 0.f, GVH = 0.f, GNV = 0.f, gO = 0.f, gLin[3], gLd[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float F = F0[c] + (1.f - F0[c]) * fc;
            const float f = (1.f - mt) * av[c] * kInvPi + spec_t * F;
            const float Lmix = (1.f - O) * Ld[c] + Lin[c];
            const float gam = sc * gov[c] * NdotL;
            const float u = gam * Lmix;
            ga[c] += u * ((1.f - mt) * kInvPi + spec_t * (1.f - fc) * mt);
            gm += u * (-av[c] * kInvPi + spec_t * (1.f - fc) * (-0.08f * a.specular + av[c]));
            gr += u * dspec_dr * F;
            GN += u * F * Gc * dD_dNH;
            GS += u * F * Gc * dD_ds2;
            GVH += u * spec_t * (1.f - F0[c]) * (-5.f * x2 * x2);
            if (!vclamp) GNV += u * F * D * G1L / (4.f * NdotL) * (-(1.f - kk) / (gvv * gvv));
            gO += -gam * f * Ld[c];
            gLin[c] = gam * f;
            gLd[c] = gam * f * (1.f - O);
        }
        // ---- scatter: probe texels (folded through the border rule) and env ----
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            // a zero weight (an empty slot of a radius search, or a probe
            // other than the one a snapped point sits on) scatters nothing
            if (k < a.K && W[k] != 0.f) {
                gW[k] += gO * tk[k].w + gLin[0] * tk[k].x + gLin[1] * tk[k].y + gLin[2] * tk[k].z;
                const float Wk = W[k];
                const float q[4] = {w00, w10, w01, w11};
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    int si, sj;
                    oct_wrap(a.R, i0 - 1 + (qq & 1), j0 - 1 + (qq >> 1), si, sj);
                    const float c = Wk * q[qq];
                    atomicAdd(a.g_maps + ((int64_t)pid[k] * a.R + sj) * a.R + si,
                              make_float4(gLin[0] * c, gLin[1] * c, gLin[2] * c, gO * c));
                }
            }
        }
#pragma unroll
        for (int qq = 0; qq < 4; ++qq)
            atomicAdd(a.genv4 + ei[qq] / 3, make_float4(gLd[0] * ew[qq], gLd[1] * ew[qq], gLd[2] * ew[qq], 0.f));
        // ---- d/dw ---------------------------------------------------------------
        // octahedral coordinates: uv = (p + 1)/2, p = w.xy/|w|_1 (folded below)
        float gw[3];
        {
            const float gs_ = gO * ps.w + gLin[0] * ps.x + gLin[1] * ps.y + gLin[2] * ps.z;
            const float gt_ = gO * pt.w + gLin[0] * pt.x + gLin[1] * pt.y + gLin[2] * pt.z;
            const float gu = gs_ * Rf, gvv2 = gt_ * Rf;  // d/d(uv)
            const float ax_ = fabsf(w.x), ay_ = fabsf(w.y), az_ = fabsf(w.z);
            const float l1 = ax_ + ay_ + az_, il2 = 1.f / (l1 * l1);
            const float sx = w.x >= 0.f ? 1.f : -1.f, sy = w.y >= 0.f ? 1.f : -1.f, sz = w.z >= 0.f ? 1.f : -1.f;
            const float dpx[3] = {(l1 - ax_) * il2, -w.x * sy * il2, -w.x * sz * il2};
            const float dpy[3] = {-w.y * sx * il2, (l1 - ay_) * il2, -w.y * sz * il2};
            if (w.z < 0.f) {
                const float px = w.x / l1, py = w.y / l1;
                const float spx = px >= 0.f ? 1.f : -1.f, spy = py >= 0.f ? 1.f : -1.f;
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    gw[c] = 0.5f * (gu * (-spy * dpy[c] * spx) + gvv2 * (-spx * dpx[c] * spy));
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) gw[c] = 0.5f * (gu * dpx[c] + gvv2 * dpy[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int j = 0; j < 3; ++j) gw[j] += gLd[c] * (dLs[c] * dsw[j] + dLt[c] * dtw[j]);
        // BRDF geometry through h, and directly through n
        const float hh[3] = {h.x, h.y, h.z}, nn[3] = {n.x, n.y, n.z}, vv[3] = {wo.x, wo.y, wo.z};
        float gh[3], gnd[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            gh[j] = GN * nn[j] + GS * 2.f * (hh[j] - NdotH * nn[j]) + GVH * vv[j];
            gnd[j] = GN * hh[j] + GS * 2.f * (nn[j] - NdotH * hh[j]) + GNV * vv[j];
        }
        if (hl > 1e-30f) {
            const float hg = hh[0] * gh[0] + hh[1] * gh[1] + hh[2] * gh[2];
#pragma unroll
            for (int j = 0; j < 3; ++j) gw[j] += (gh[j] - hg * hh[j]) / hl;
        }
        // w = l.x t(n) + l.y b(n) + l.z n
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float v = l.z * gw[j] + gnd[j];
#pragma unroll
            for (int c = 0; c < 3; ++c) v += l.x * gw[c] * dt[c][j] + l.y * gw[c] * db[c][j];
            gn[j] += v;
        }
    }
    // blend weights W_k = w_s w_b / sum (Eq. 5-6) over the probes found (the
    // nonzero W: a found probe's weight is at least 0.01 w_s / sum): w_b moves
    // with the normal. A one-hot W (a point sitting on its nearest probe, or
    // a radius search that found one probe) and an all-zero one (none found)
    // do not depend on it; then W[1] == 0.
    const bool snapped = a.K > 1 && W[1] == 0.f;
    if (a.K > 1 && !snapped) {
        const float3 xp = load3(a.x, m);
        float U = 0.f, ws[KMAX], gdot = 0.f;
        float3 dh[KMAX];
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            ws[k] = 0.f;
            dh[k] = f3(0.f, 0.f, 0.f);
            if (k < a.K && W[k] != 0.f) {
                const float3 d = load3(a.probe_pos, pid[k]) - xp;
                const float dl = sqrtf(dot3(d, d));
                ws[k] = 1.f / dl;
                dh[k] = (1.f / dl) * d;
                U += ws[k] * (0.5f * (1.f + dot3(dh[k], n)) + 0.01f);
                gdot += gW[k] * W[k];
            }
        }
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            if (k < a.K && W[k] != 0.f) {
                const float gu = (gW[k] - gdot) / U;
                gn[0] += gu * ws[k] * 0.5f * dh[k].x;
                gn[1] += gu * ws[k] * 0.5f * dh[k].y;
                gn[2] += gu * ws[k] * 0.5f * dh[k].z;
            }
        }
    }
    // through n = n_raw / |n_raw|
    const float ng = gn[0] * n.x + gn[1] * n.y + gn[2] * n.z;
    a.g_normal[3 * m] = (gn[0] - ng * n.x) / nl;
    a.g_normal[3 * m + 1] = (gn[1] - ng * n.y) / nl;
    a.g_normal[3 * m + 2] = (gn[2] - ng * n.z) / nl;
    a.g_albedo[3 * m] = ga[0];
    a.g_albedo[3 * m + 1] = ga[1];
    a.g_albedo[3 * m + 2] = ga[2];
    a.g_rough[m] = gr;
    a.g_metal[m] = gm;
}

// ---------------------------------------------------------------------------
// The adjoint with eight points a CTA, one warp a point.
//
// A direction's footprint lies at the same place of every probe's map, so a
// point's map gradient is one image: G[t] = sum over its directions of the
// bilinear weight of texel t times (dL/dL_in, dL/dO), and probe k receives
// W_k G while dL/dW_k = <G, map_k>. So each warp
//  - blends the texels that its directions touch once (as in
//    point_blend.cuh), here for the CTA's eight points together: a texel of
//    each of their probes is read once and added to every point that has it;
//  - takes its directions 32 at a time, reading and scattering four texels
//    of its own two images in shared memory, never the atlas;
//  - and the CTA adds each probe's sum over the points to the gradient, one
//    vector atomic a texel, reading the map once more for the eight products.
// Points come grouped by nearest probe, so the eight share most of their
// probes. Per point and direction the former kernel made K 4 gathers and K 4
// vector atomics in L2, which bound it.
// The scatter takes two directions a step, half a warp each: a lane owns one
// corner and one component, so nothing collides within a footprint; pairs
// whose footprints touch are taken one after the other. Every sum of a point
// keeps one order whatever points share its CTA (probes by index, texels by
// place), so a point's gradients are the same on every run.
// Bound: instruction issue and latency (16 warps an SM, 8,000 instructions a
// point at S = 128). 418,111 points, K = 8, S = 128: 12.4 -> 6.8 ms.
// ---------------------------------------------------------------------------
constexpr int kAdjPts = 8;

struct AdjSmem {
    size_t dirs, map, grad, rec, wu, gwu, pid, slot, mark, list, wrap, total;
};
__host__ __device__ inline AdjSmem adj_smem(int R, int S, int K)
{
    const size_t t = (size_t)point_texels(R), u = (size_t)kAdjPts * K;
    AdjSmem L;
    size_t o = 0;
    L.dirs = o; o += 16 * (size_t)S;
    L.map = o;  o += 16 * t * kAdjPts;
    L.grad = o; o += 16 * t * kAdjPts;
    L.rec = o;  o += 64 * 32 * kAdjPts;
    L.wu = o;   o += 4 * u * kAdjPts;
    L.gwu = o;  o += 4 * u * kAdjPts;
    L.pid = o;  o += 4 * u;
    L.slot = o; o += 4 * u;
    L.mark = o; o += 4 * (size_t)(point_words(R) + 1);
    L.list = o; o += 2 * t;
    L.wrap = o; o += 2 * t;
    L.total = (o + 15) & ~(size_t)15;
    return L;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int DT>
__global__ void __launch_bounds__(kAdjPts * 32, 2) adjoint_tile_kernel(const AdjK a)
{
    using TX = Texel<DT>;
    extern __shared__ __align__(16) char s_raw[];
    __shared__ int s_offs[kAdjPts][32];
    __shared__ uint32_t s_present[kAdjPts];
    __shared__ int16_t s_place[kAdjPts * 32];
    const AdjSmem L = adj_smem(a.R, a.S, a.K);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
    const unsigned full = 0xffffffffu;
    const int RS = a.R + 2, T = RS * RS, words = point_words(a.R), K = a.K;
    float4* s_dirs = reinterpret_cast<float4*>(s_raw + L.dirs);
    float4* s_map = reinterpret_cast<float4*>(s_raw + L.map);    // [8][T]
    float4* s_grad = reinterpret_cast<float4*>(s_raw + L.grad);  // [8][T]
    float4* rec = reinterpret_cast<float4*>(s_raw + L.rec) + warp * 128;  // this warp's 32 directions x 4 corners
    float* s_wu = reinterpret_cast<float*>(s_raw + L.wu);        // [U][8] weight of probe u for point p
    const float4* s_wu4 = reinterpret_cast<const float4*>(s_wu);
    float* s_gwu = reinterpret_cast<float*>(s_raw + L.gwu);      // [U][8] dL/dW
    int32_t* s_pid = reinterpret_cast<int32_t*>(s_raw + L.pid);  // [U] the points' probes, by index
    int32_t* s_slot = reinterpret_cast<int32_t*>(s_raw + L.slot);  // [8][K] (probe, then its place in s_pid)
    uint32_t* s_mark = reinterpret_cast<uint32_t*>(s_raw + L.mark);
    uint16_t* s_list = reinterpret_cast<uint16_t*>(s_raw + L.list);
    uint16_t* s_wrap = reinterpret_cast<uint16_t*>(s_raw + L.wrap);
    int* s_off = s_offs[warp];
    // ---- tables, once for all of this CTA's tiles ---------------------------
    for (int i = tid; i < a.S; i += blockDim.x) s_dirs[i] = a.dirs[i];
    for (int t = tid; t < T; t += blockDim.x) {
        int si, sj;
        oct_wrap(a.R, t % RS - 1, t / RS - 1, si, sj);
        s_wrap[t] = (uint16_t)(sj * a.R + si);
    }
    // a CTA's tiles lie next to one another in the grouped order: they share
    // probes, and other CTAs add to other texels
    const int64_t tiles = (a.M + kAdjPts - 1) / kAdjPts;
    const int64_t tile_end = tiles * (blockIdx.x + 1) / gridDim.x;
    for (int64_t tile = tiles * blockIdx.x / gridDim.x; tile < tile_end; ++tile) {
    const int64_t pos = tile * kAdjPts + warp;  // position in the grouped order
    const bool active = pos < a.M;
    const int64_t m = active ? __ldg(a.perm + pos) : 0;

    // ---- the union of the points' probes, in index order --------------------
    for (int i = tid; i < kAdjPts * kAdjPts * K; i += blockDim.x) s_wu[i] = 0.f;
    for (int w = tid; w <= words; w += blockDim.x) s_mark[w] = 0u;
    if (tid < kAdjPts) s_present[tid] = 0u;
    // a zero weight (an empty slot of a radius search, or a probe other than
    // the one a snapped point sits on) takes and gives nothing
    const float Wl = active && lane < K ? __ldg(a.w + m * K + lane) : 0.f;
    const int32_t idl = active && lane < K ? __ldg(a.idx + m * K + lane) : 0;
    if (lane < K) s_slot[warp * K + lane] = Wl != 0.f ? idl : INT32_MAX;
    __syncthreads();
    // the number of entries with a smaller probe is the same for all entries
    // of one probe and differs between probes: its place among 8 K, of which
    // the ones present are then counted (four threads an entry)
    for (int e0 = 0; e0 < kAdjPts * K; e0 += kAdjPts * 8) {
        const int e = e0 + (tid >> 2);
        const int32_t id = e < kAdjPts * K ? s_slot[e] : INT32_MAX;
        int below = 0;
        for (int j = tid & 3; j < kAdjPts * K; j += 4) below += s_slot[j] < id ? 1 : 0;
        below += __shfl_xor_sync(full, below, 1);
        below += __shfl_xor_sync(full, below, 2);
        if ((tid & 3) == 0 && id != INT32_MAX) {
            s_place[e] = (int16_t)below;
            atomicOr(&s_present[below >> 5], 1u << (below & 31));
        }
    }
    __syncthreads();
    int my_slot = -1, U = 0;
    {
        const int place = lane < K && Wl != 0.f ? s_place[warp * K + lane] : -1;
#pragma unroll
        for (int w = 0; w < kAdjPts; ++w) {
            const uint32_t b = s_present[w];
            if (place >> 5 == w) my_slot = U + __popc(b & ((1u << (place & 31)) - 1u));
            U += __popc(b);
        }
        if (place < 0) my_slot = -1;
    }
    if (my_slot >= 0) s_pid[my_slot] = idl;
    if (my_slot >= 0) s_wu[my_slot * kAdjPts + warp] = Wl;

    // ---- the point ----------------------------------------------------------
    const float3 nr = load3(a.n, m);
    const float nl = sqrtf(dot3(nr, nr));
    const float3 n = f3(nr.x / nl, nr.y / nl, nr.z / nl);
    float3 tt, bb;
    onb(n, tt, bb);
    const float3 wo = load3(a.wo, m);
    const float3 alb = load3(a.albedo, m);
    const float r = __ldg(a.rough + m), mt = __ldg(a.metal + m);
    const float3 go = load3(a.grad_out, m);
    if (a.status && active && lane == 0 &&
        !isfinite(go.x + go.y + go.z + alb.x + alb.y + alb.z + r + mt + wo.x + wo.y + wo.z))
        atomicOr(a.status, SOP_DEVSTAT_NONFINITE);
    const float Rf = (float)a.R;
    const auto world = [&](const float4 l) {
        return f3(fmaf(l.x, tt.x, fmaf(l.y, bb.x, l.z * n.x)), fmaf(l.x, tt.y, fmaf(l.y, bb.y, l.z * n.y)),
                  fmaf(l.x, tt.z, fmaf(l.y, bb.z, l.z * n.z)));
    };
    PointSmem sm;
    sm.map = s_map + (size_t)warp * T;
    sm.mark = s_mark;
    sm.list = s_list;
    if (active)
        for (int i = lane; i < a.S; i += 32) point_mark(sm, oct_foot(world(s_dirs[i]), Rf, a.R).off, RS);
    __syncthreads();

    // ---- the blended texels of all eight points ------------------------------
    // (each warp lists its share of the mark words)
    int nt = 0;
    for (int w0 = 0; w0 < words; w0 += 32) {
        const uint32_t mk = w0 + lane < words ? s_mark[w0 + lane] : 0u;
        int upto = __popc(mk);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(full, upto, o);
            if (lane >= o) upto += v;
        }
        for (int w = warp; w < 32 && w0 + w < words; w += kAdjPts) {
            const uint32_t b = __shfl_sync(full, mk, w);
            const int base = nt + __shfl_sync(full, upto, w) - __popc(b);
            if ((b >> lane) & 1u) s_list[base + __popc(b & ((1u << lane) - 1u))] = (uint16_t)((w0 + w) * 32 + lane);
        }
        nt += __shfl_sync(full, upto, 31);
    }
    __syncthreads();
    const typename TX::raw* atlas = reinterpret_cast<const typename TX::raw*>(a.rgbo);
    for (int j = tid; j < nt; j += blockDim.x) {
        const uint32_t t = s_list[j];
        float4 v[kAdjPts];
#pragma unroll
        for (int p = 0; p < kAdjPts; ++p) v[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int u0 = 0; u0 < U; u0 += 4) {
            float4 x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                x[q] = TX::load(atlas + ((uint32_t)s_pid[min(u0 + q, U - 1)] * (uint32_t)T + t));
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (u0 + q >= U) break;
                const float4 wa = s_wu4[2 * (u0 + q)], wb = s_wu4[2 * (u0 + q) + 1];
                const float wp[kAdjPts] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
                for (int p = 0; p < kAdjPts; ++p)
                    if (wp[p] != 0.f) {
                        v[p].x = fmaf(wp[p], x[q].x, v[p].x);
                        v[p].y = fmaf(wp[p], x[q].y, v[p].y);
                        v[p].z = fmaf(wp[p], x[q].z, v[p].z);
                        v[p].w = fmaf(wp[p], x[q].w, v[p].w);
                    }
            }
        }
#pragma unroll
        for (int p = 0; p < kAdjPts; ++p) {
            s_map[(size_t)p * T + t] = v[p];
            s_grad[(size_t)p * T + t] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __syncthreads();

    // ---- the directions --------------------------------------------------------
    const float al = r * r, a2 = al * al, kk = (r + 1.f) * (r + 1.f) * 0.125f;
    const float NdotVraw = dot3(n, wo);
    const bool vclamp = NdotVraw < 1e-4f;
    const float NdotV = vclamp ? 1e-4f : NdotVraw;
    const float gvv = NdotV * (1.f - kk) + kk;
    const float G1V = NdotV / gvv;
    const float i4nv = 1.f / (4.f * NdotV);
    // d spec / d r through G, and d spec / d NdotV, up to the per-direction factors
    const float cr0 = (r + 1.f) * 0.25f * i4nv, cr1 = -NdotV * (1.f - NdotV) / (gvv * gvv);
    const float cnv = vclamp ? 0.f : -0.25f * (1.f - kk) / (gvv * gvv);
    const float G1Vn = G1V * i4nv, r3 = 4.f * r * r * r;
    const float f0d = 0.08f * a.specular * (1.f - mt);
    const float F0[3] = {f0d + alb.x * mt, f0d + alb.y * mt, f0d + alb.z * mt};
    const float av[3] = {alb.x, alb.y, alb.z};
    const float sc = 2.f * kPi / (float)a.S;
    const float gov[3] = {sc * go.x, sc * go.y, sc * go.z};
    const float kd0 = (1.f - mt) * kInvPi;
    float ga[3] = {0.f, 0.f, 0.f}, gr = 0.f, gm = 0.f;
    // dL/dn: sums of l.z dL/dw + (direct part), l.x dL/dw and l.y dL/dw; the
    // last two go through the frame's derivatives after the loop
    float gn[3] = {0.f, 0.f, 0.f}, gt[3] = {0.f, 0.f, 0.f}, gb[3] = {0.f, 0.f, 0.f};
    float* grad = reinterpret_cast<float*>(s_grad + (size_t)warp * T);
    for (int i0 = 0; active && i0 < a.S; i0 += 32) {
        const int i = i0 + lane;
        const bool on = i < a.S;
        const float4 l = s_dirs[on ? i : 0];
        const float3 w = world(l);
        const float NdotL = l.z;
        const Foot ft = oct_foot(w, Rf, a.R);
        const float fu = ft.fu, fv = ft.fv;
        const float w00 = (1.f - fu) * (1.f - fv), w10 = fu * (1.f - fv), w01 = (1.f - fu) * fv, w11 = fu * fv;
        float gO = 0.f, gLin[3] = {0.f, 0.f, 0.f};
        if (on) {
            // ---- environment and its direction derivative -------------------
            const float rho2 = w.x * w.x + w.y * w.y, rho = sqrtf(rho2);
            const float th = atan2f(rho, w.z), ph = atan2f(w.y, w.x);
            const float es = (ph + kPi) * kInv2Pi * a.We - 0.5f, et = th * kInvPi * a.He - 0.5f;
            const float fes = floorf(es), fet = floorf(et);
            const float ea = es - fes, eb = et - fet;
            int c0 = (int)fes;
            c0 = c0 < 0 ? c0 + a.We : c0;
            c0 = min(max(c0, 0), a.We - 1);
            const int c1 = c0 + 1 == a.We ? 0 : c0 + 1;
            const int r0 = min(max((int)fet, 0), a.He - 1), r1 = min(max((int)fet + 1, 0), a.He - 1);
            const int ei[4] = {r0 * a.We + c0, r0 * a.We + c1, r1 * a.We + c0, r1 * a.We + c1};
            float e4[4][3];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) e4[q][c] = __ldg(a.env + 3 * (int64_t)ei[q] + c);
            const float ew[4] = {(1.f - ea) * (1.f - eb), ea * (1.f - eb), (1.f - ea) * eb, ea * eb};
            // ---- probe terms --------------------------------------------------
            const float4 t00 = sm.map[ft.off], t10 = sm.map[ft.off + 1], t01 = sm.map[ft.off + RS],
                         t11 = sm.map[ft.off + RS + 1];
            const float O = w00 * t00.w + w10 * t10.w + w01 * t01.w + w11 * t11.w;
            const float Lin[3] = {w00 * t00.x + w10 * t10.x + w01 * t01.x + w11 * t11.x,
                                  w00 * t00.y + w10 * t10.y + w01 * t01.y + w11 * t11.y,
                                  w00 * t00.z + w10 * t10.z + w01 * t01.z + w11 * t11.z};
            // ---- BRDF -----------------------------------------------------------
            const float3 hv = w + wo;
            const float hl2 = dot3(hv, hv);
            const float ihl = hl2 > 1e-30f ? 1.f / sqrtf(hl2) : 0.f;
            const float3 h = hl2 > 1e-30f ? ihl * hv : n;
            const float NdotH = dot3(n, h), VdotH = dot3(wo, h);
            const float3 cr = cross3(n, h);
            const float sin2 = dot3(cr, cr);
            const float den = NdotH * NdotH * a2 + sin2, iden = 1.f / den, igl = 1.f / (NdotL * (1.f - kk) + kk);
            const float ip2 = kInvPi * iden * iden, D = a2 * ip2, Gc = igl * G1Vn, spec_t = D * Gc;
            const float x1 = 1.f - VdotH, x2 = x1 * x1, fc = x2 * x2 * x1;
            const float dspec_dr = (den - 2.f * a2 * NdotH * NdotH) * iden * ip2 * r3 * Gc +
                                   D * cr0 * igl * (cr1 - (1.f - NdotL) * igl * G1V);
            float gLd[3], SF = 0.f, SV = 0.f;
            const float s1 = spec_t * (1.f - fc);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float Ld = ew[0] * e4[0][c] + ew[1] * e4[1][c] + ew[2] * e4[2][c] + ew[3] * e4[3][c];
                const float F = F0[c] + (1.f - F0[c]) * fc;
                const float f = kd0 * av[c] + spec_t * F;
                const float gam = gov[c] * NdotL, u = gam * ((1.f - O) * Ld + Lin[c]);
                ga[c] += u * (kd0 + s1 * mt);
                gm += u * (-av[c] * kInvPi + s1 * (-0.08f * a.specular + av[c]));
                SF += u * F;
                SV += u * (1.f - F0[c]);
                gLin[c] = gam * f;
                gLd[c] = gLin[c] * (1.f - O);
                gO -= gLin[c] * Ld;
            }
            gr += SF * dspec_dr;
            // dL/d(n.h), dL/d|n x h|^2, dL/d(v.h), dL/d(n.v). (-2 a2 / (pi den^3)
            // as -2 D / den: den is r^4 at the mirror direction, whose inverse
            // cube alone leaves float32 below r = 5.6e-4)
            const float GS = SF * Gc * (-2.f * (D * iden)), GN = 2.f * a2 * NdotH * GS;
            const float GVH = SV * spec_t * (-5.f * x2 * x2), GNV = SF * D * igl * cnv;
            // ---- scatter: environment -------------------------------------------
#pragma unroll
            for (int q = 0; q < 4; ++q)
                atomicAdd(a.genv4 + ei[q], make_float4(gLd[0] * ew[q], gLd[1] * ew[q], gLd[2] * ew[q], 0.f));
            // ---- d/dw -------------------------------------------------------------
            // map coordinates: d/ds = (1-fv)(t10-t00) + fv(t11-t01), d/dt = (1-fu)(t01-t00) + fu(t11-t10),
            // and uv = (p + 1)/2, p = w.xy/|w|_1 (folded below)
            const auto dotg = [&](const float4 p) { return gO * p.w + gLin[0] * p.x + gLin[1] * p.y + gLin[2] * p.z; };
            const float4 d10 = make_float4(t10.x - t00.x, t10.y - t00.y, t10.z - t00.z, t10.w - t00.w);
            const float4 d11 = make_float4(t11.x - t01.x, t11.y - t01.y, t11.z - t01.z, t11.w - t01.w);
            const float4 e01 = make_float4(t01.x - t00.x, t01.y - t00.y, t01.z - t00.z, t01.w - t00.w);
            const float4 e11 = make_float4(t11.x - t10.x, t11.y - t10.y, t11.z - t10.z, t11.w - t10.w);
            const float gu = ((1.f - fv) * dotg(d10) + fv * dotg(d11)) * Rf;
            const float gv = ((1.f - fu) * dotg(e01) + fu * dotg(e11)) * Rf;
            const float ax_ = fabsf(w.x), ay_ = fabsf(w.y), az_ = fabsf(w.z);
            const float l1 = ax_ + ay_ + az_, il2 = 1.f / (l1 * l1);
            const float sx = w.x >= 0.f ? 1.f : -1.f, sy = w.y >= 0.f ? 1.f : -1.f, sz = w.z >= 0.f ? 1.f : -1.f;
            const float fold = w.z < 0.f ? -sx * sy : 0.f;
            const float px = 0.5f * il2 * (w.z < 0.f ? fold * gv : gu), py = 0.5f * il2 * (w.z < 0.f ? fold * gu : gv);
            // dp.x = (l1 - |x|, -x sy, -x sz) / l1^2, dp.y = (-y sx, l1 - |y|, -y sz) / l1^2
            float gw[3] = {px * (l1 - ax_) - py * w.y * sx, py * (l1 - ay_) - px * w.x * sy,
                           -(px * w.x + py * w.y) * sz};
            // environment coordinates: ds/dw, dt/dw
            if (rho2 > 0.f) {
                float gs = 0.f, gte = 0.f;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    gs += gLd[c] * ((1.f - eb) * (e4[1][c] - e4[0][c]) + eb * (e4[3][c] - e4[2][c]));
                    gte += gLd[c] * ((1.f - ea) * (e4[2][c] - e4[0][c]) + ea * (e4[3][c] - e4[1][c]));
                }
                const float ks = gs * (a.We * kInv2Pi / rho2);
                const float kt = gte * (a.He * kInvPi / (rho2 + w.z * w.z)), kz = kt * w.z / rho;
                gw[0] += kz * w.x - ks * w.y;
                gw[1] += kz * w.y + ks * w.x;
                gw[2] -= kt * rho;
            }
            // BRDF geometry through h, and directly through n
            const float hh[3] = {h.x, h.y, h.z}, nn[3] = {n.x, n.y, n.z}, vv[3] = {wo.x, wo.y, wo.z};
            float gh[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) gh[j] = GN * nn[j] + 2.f * GS * (hh[j] - NdotH * nn[j]) + GVH * vv[j];
            const float hg = hh[0] * gh[0] + hh[1] * gh[1] + hh[2] * gh[2];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                gw[j] += (gh[j] - hg * hh[j]) * ihl;
                // w = l.x t(n) + l.y b(n) + l.z n
                gn[j] += l.z * gw[j] + (GN * hh[j] + 2.f * GS * (nn[j] - NdotH * hh[j]) + GNV * vv[j]);
                gt[j] += l.x * gw[j];
                gb[j] += l.y * gw[j];
            }
        }
        // ---- scatter: this warp's gradient image, two directions a step ------
        // (each lane lays out its direction's 4 corners x 4 components)
        float4* rv = rec + 4 * lane;
        rv[0] = make_float4(w00 * gLin[0], w00 * gLin[1], w00 * gLin[2], w00 * gO);
        rv[1] = make_float4(w10 * gLin[0], w10 * gLin[1], w10 * gLin[2], w10 * gO);
        rv[2] = make_float4(w01 * gLin[0], w01 * gLin[1], w01 * gLin[2], w01 * gO);
        rv[3] = make_float4(w11 * gLin[0], w11 * gLin[1], w11 * gLin[2], w11 * gO);
        s_off[lane] = ft.off;
        // steps whose two footprints share a texel (bases at most one apart)
        const int other = __shfl_xor_sync(full, ft.off, 16), dd = abs(other - ft.off);
        const unsigned touch = __ballot_sync(full, dd <= 1 || (dd >= RS - 1 && dd <= RS + 1));
        __syncwarp();
        const float* val = reinterpret_cast<const float*>(rec) + (lane & 15);
        float* at0 = grad + ((lane & 3) + 4 * (((lane >> 2) & 1) + ((lane >> 3) & 1) * RS));
        const int sh = lane & 16, steps = min(16, a.S - i0);
        if ((touch & ((1u << steps) - 1u)) == 0u) {
#pragma unroll 4
            for (int st = 0; st < steps; ++st) {
                float* at = at0 + 4 * s_off[st + sh];
                *at += val[16 * (st + sh)];
                __syncwarp();
            }
        } else {
            for (int st = 0; st < steps; ++st) {
                float* at = at0 + 4 * s_off[st + sh];
                const float g = val[16 * (st + sh)];
                if (sh == 0 || !((touch >> st) & 1u)) *at += g;
                __syncwarp();
                if (sh != 0 && ((touch >> st) & 1u)) *at += g;
                __syncwarp();
            }
        }
    }
    __syncthreads();

    // ---- to the probes: their gradients, and the eight products ---------------
    uint32_t col0 = 0u;  // this lane's column of the first 32 mark words
    for (int w = 0; w < 32 && w < words; ++w) col0 |= ((s_mark[w] >> lane) & 1u) << w;
    for (int u = warp; u < U; u += kAdjPts) {
        float wp[kAdjPts], dot[kAdjPts];
#pragma unroll
        for (int p = 0; p < kAdjPts; ++p) {
            wp[p] = s_wu[u * kAdjPts + p];
            dot[p] = 0.f;
        }
        const int32_t pid = s_pid[u];
        float4* gmap = a.g_maps + (int64_t)pid * a.R * a.R;
        // a lane takes the marked texels of its own column, t mod 32, in
        // order (not the list's: the order of a point's sum is its own)
        for (int w0 = 0; w0 < words; w0 += 32) {
            uint32_t col = w0 == 0 ? col0 : 0u;
            if (w0 > 0)
                for (int w = 0; w < 32 && w0 + w < words; ++w) col |= ((s_mark[w0 + w] >> lane) & 1u) << w;
            while (col) {
                int t[2];
                float4 x[2];
                const bool two = (col & (col - 1)) != 0u;
                t[0] = (w0 + __ffs(col) - 1) * 32 + lane;
                col &= col - 1;
                t[1] = two ? (w0 + __ffs(col) - 1) * 32 + lane : t[0];
                col &= col - 1;
                x[0] = TX::load(atlas + ((uint32_t)pid * (uint32_t)T + (uint32_t)t[0]));
                if (two) x[1] = TX::load(atlas + ((uint32_t)pid * (uint32_t)T + (uint32_t)t[1]));
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    if (q == 1 && !two) break;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int p = 0; p < kAdjPts; ++p)
                        if (wp[p] != 0.f) {
                            const float4 g = s_grad[(size_t)p * T + t[q]];
                            v.x = fmaf(wp[p], g.x, v.x);
                            v.y = fmaf(wp[p], g.y, v.y);
                            v.z = fmaf(wp[p], g.z, v.z);
                            v.w = fmaf(wp[p], g.w, v.w);
                            dot[p] = fmaf(g.x, x[q].x, fmaf(g.y, x[q].y, fmaf(g.z, x[q].z, fmaf(g.w, x[q].w, dot[p]))));
                        }
                    if (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f) atomicAdd(gmap + s_wrap[t[q]], v);
                }
            }
            __syncwarp();
        }
#pragma unroll
        for (int p = 0; p < kAdjPts; ++p) {
            if (wp[p] == 0.f) continue;
            const float v = warp_sum(dot[p]);
            if (lane == 0) s_gwu[u * kAdjPts + p] = v;
        }
    }
    __syncthreads();
    if (!active) continue;  // (only in the last tile)

    // ---- the point's own gradients ---------------------------------------------
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        ga[c] = warp_sum(ga[c]);
        gn[c] = warp_sum(gn[c]);
    }
    gr = warp_sum(gr);
    gm = warp_sum(gm);
    {
        // frame derivatives (Duff et al. 2017): dt/dn and db/dn, row = component
        const float sg = n.z >= 0.f ? 1.f : -1.f, aa = -1.f / (sg + n.z), a2n = aa * aa;
        const float dt[3][3] = {{2.f * sg * n.x * aa, 0.f, sg * n.x * n.x * a2n},
                                {sg * n.y * aa, sg * n.x * aa, sg * n.x * n.y * a2n},
                                {-sg, 0.f, 0.f}};
        const float db[3][3] = {{n.y * aa, n.x * aa, n.x * n.y * a2n}, {0.f, 2.f * n.y * aa, n.y * n.y * a2n},
                                {0.f, -1.f, 0.f}};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            gt[c] = warp_sum(gt[c]);
            gb[c] = warp_sum(gb[c]);
#pragma unroll
            for (int j = 0; j < 3; ++j) gn[j] += gt[c] * dt[c][j] + gb[c] * db[c][j];
        }
    }
    // blend weights W_k = w_s w_b / sum (Eq. 5-6) over the probes found (the
    // nonzero W: a found probe's weight is at least 0.01 w_s / sum): w_b moves
    // with the normal. A one-hot W (a point sitting on its nearest probe, or
    // a radius search that found one probe) and an all-zero one (none found)
    // do not depend on it; then W[1] == 0. Lane k takes probe k.
    if (K > 1 && __shfl_sync(full, Wl, 1) != 0.f) {
        float U_ = 0.f, ws = 0.f, gw = 0.f;
        float3 dh = f3(0.f, 0.f, 0.f);
        if (my_slot >= 0) {
            const float3 d = load3(a.probe_pos, idl) - load3(a.x, m);
            const float dl = sqrtf(dot3(d, d));
            ws = 1.f / dl;
            dh = (1.f / dl) * d;
            U_ = ws * (0.5f * (1.f + dot3(dh, n)) + 0.01f);
            gw = s_gwu[my_slot * kAdjPts + warp];
        }
        U_ = warp_sum(U_);
        const float gdot = warp_sum(gw * Wl);
        const float gu = my_slot >= 0 ? (gw - gdot) / U_ * ws * 0.5f : 0.f;
        gn[0] += warp_sum(gu * dh.x);
        gn[1] += warp_sum(gu * dh.y);
        gn[2] += warp_sum(gu * dh.z);
    }
    // through n = n_raw / |n_raw|
    const float ng = gn[0] * n.x + gn[1] * n.y + gn[2] * n.z;
    if (lane < 3) {
        const float gnl = lane == 0 ? gn[0] : (lane == 1 ? gn[1] : gn[2]);
        const float nn = lane == 0 ? n.x : (lane == 1 ? n.y : n.z);
        a.g_normal[3 * m + lane] = (gnl - ng * nn) / nl;
        a.g_albedo[3 * m + lane] = lane == 0 ? ga[0] : (lane == 1 ? ga[1] : ga[2]);
    }
    if (lane == 0) {
        a.g_rough[m] = gr;
        a.g_metal[m] = gm;
    }
    }  // next tile
}
// ---- grouping of the points by nearest probe (counting sort) -----------------
__global__ void perm_count_kernel(const int32_t* __restrict__ idx, int32_t K, int64_t M, int32_t* __restrict__ bucket)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m < M) atomicAdd(bucket + idx[m * K], 1);
}

__global__ void __launch_bounds__(1024) perm_scan_kernel(int32_t* __restrict__ bucket, int32_t P)
{
    __shared__ int32_t s_part[1024];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int chunk = (P + nt - 1) / nt, c0 = tid * chunk, c1 = min(P, c0 + chunk);
    int32_t sum = 0;
    for (int c = c0; c < c1; ++c) sum += bucket[c];
    s_part[tid] = sum;
    __syncthreads();
    for (int off = 1; off < nt; off <<= 1) {
        const int32_t v = tid >= off ? s_part[tid - off] : 0;
        __syncthreads();
        s_part[tid] += v;
        __syncthreads();
    }
    int32_t run = s_part[tid] - sum;
    for (int c = c0; c < c1; ++c) {
        const int32_t v = bucket[c];
        bucket[c] = run;
        run += v;
    }
}

__global__ void perm_fill_kernel(const int32_t* __restrict__ idx, int32_t K, int64_t M, int32_t* __restrict__ bucket,
                                 int32_t* __restrict__ perm)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m < M) perm[atomicAdd(bucket + idx[m * K], 1)] = (int32_t)m;
}

__global__ void env_fold_kernel(const float4* __restrict__ genv4, int64_t n, float* __restrict__ g_env)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const float4 v = genv4[t];
    g_env[3 * t] += v.x;
    g_env[3 * t + 1] += v.y;
    g_env[3 * t + 2] += v.z;
}

template <int DT, int KMAX>
static cudaError_t adjoint_launch(const AdjK& k, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * (size_t)k.S;
    auto fn = adjoint_kernel<DT, KMAX>;
    if (const cudaError_t e = allow_smem(fn, smem); e != cudaSuccess) return e;
    fn<<<(unsigned)((k.M + 127) / 128), 128, smem, s>>>(k);
    return cudaGetLastError();
}

// Which kernel: the tile kernel has a cost a point for its texels (union,
// blend, flush: (R+2)^2 of them stored) and a smaller one a direction than
// the thread-per-point kernel, whose cost is its S K gathers and atomics.
// Measured at R = 16 on 418,111 points of a view, us a call (thread / tile):
// S 128, K 8: 12,680 / 7,270; S 64, K 8: 6,760 / 5,460; S 32, K 8: 3,850 /
// 4,420; S 32, K 4: 2,220 / 3,430. R = 24, 100,000 points: S 128: 3,630 /
// 3,750, S 32: 1,120 / 2,270. So the line lies near S K = 1.5 (R+2)^2, and on
// small maps near S (K + 4) = 100 (60,000 points, R 2, K 4, S 8: 280 / 354). A
// thread takes its S directions one after the other, about 8 us each however
// few points there are, so small calls go to the tile kernel (1,000 points,
// S 128: 1,080 / 310; 8,191 points: 1,060 / 450) unless they have few
// directions: the line rises with the points, and twice as fast where an SM
// holds one CTA instead of two (16,384 points, K 4: R 8: S 16 177 / 189, S 32 229
// / 196; R 16: S 32 224 / 228, S 64 345 / 267; R 24: S 8 130 / 285, S 64 342 /
// 440).
constexpr int64_t kAdjSmall = 16384;
constexpr size_t kAdjTwoCtas = 110 * 1024;  // shared memory of two CTAs an SM
static bool adjoint_by_tile(const AdjK& k)
{
    const size_t smem = adj_smem(k.R, k.S, k.K).total;
    if (smem > kSmemMost) return false;
    const int64_t t = point_texels(k.R), sk = (int64_t)k.S * k.K;
    const int64_t least = (100 + 3 * t / 5) * (smem <= kAdjTwoCtas ? 1 : 2);
    if (k.M <= kAdjSmall) return (sk + 4 * (int64_t)k.S) * kAdjSmall >= least * k.M;
    return 2 * sk >= 3 * t && sk + 4 * (int64_t)k.S >= least;
}

template <int DT>
static cudaError_t adjoint_tile_launch(const AdjK& k, cudaStream_t s)
{
    const size_t smem = adj_smem(k.R, k.S, k.K).total;
    auto fn = adjoint_tile_kernel<DT>;
    int dev = 0, sms = 0;
    cudaError_t e = allow_smem(fn, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // two CTAs an SM (their registers' limit) where shared memory holds both
    const int64_t tiles = (k.M + kAdjPts - 1) / kAdjPts, most = (int64_t)sms * (smem <= kAdjTwoCtas ? 2 : 1);
    fn<<<(unsigned)(tiles < most ? tiles : most), kAdjPts * 32, smem, s>>>(k);
    return cudaGetLastError();
}

template <int DT>
static cudaError_t adjoint_k(const AdjK& k, cudaStream_t s)
{
    if (adjoint_by_tile(k)) return adjoint_tile_launch<DT>(k, s);
    if (k.K <= 4) return adjoint_launch<DT, 4>(k, s);
    if (k.K <= 8) return adjoint_launch<DT, 8>(k, s);
    if (k.K <= 16) return adjoint_launch<DT, 16>(k, s);
    return adjoint_launch<DT, 32>(k, s);
}

cudaError_t launch_adjoint(const QueryArgs& a, const QueryLayout& L, char* ws, cudaStream_t s)
{
    if (a.M == 0) return cudaSuccess;
    AdjK k;
    k.x = a.x;
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
    k.env = a.env;
    k.dirs = reinterpret_cast<const float4*>(ws + L.dirs);
    k.idx = reinterpret_cast<const int32_t*>(ws + L.idx);
    k.w = reinterpret_cast<const float*>(ws + L.w);
    k.probe_pos = a.probe_pos;
    k.specular = a.specular;
    k.grad_out = a.grad_out;
    k.status = status_word();
    k.g_albedo = a.g_albedo;
    k.g_rough = a.g_rough;
    k.g_metal = a.g_metal;
    k.g_normal = a.g_normal;
    k.g_env = a.g_env;
    k.g_maps = reinterpret_cast<float4*>(a.g_atlas);
    int32_t* perm = reinterpret_cast<int32_t*>(ws + L.perm);
    int32_t* bucket = reinterpret_cast<int32_t*>(ws + L.bucket);
    k.perm = perm;
    k.genv4 = reinterpret_cast<float4*>(ws + L.genv4);

    // (the buckets and the environment gradient lie next to each other)
    cudaError_t e = cudaMemsetAsync(bucket, 0, L.genv4 - L.bucket + sizeof(float4) * (size_t)a.He * a.We, s);
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)((a.M + 255) / 256);
    perm_count_kernel<<<nb, 256, 0, s>>>(k.idx, a.K, a.M, bucket);
    perm_scan_kernel<<<1, 1024, 0, s>>>(bucket, a.P);
    perm_fill_kernel<<<nb, 256, 0, s>>>(k.idx, a.K, a.M, bucket, perm);
    switch (a.rgbo_dtype) {
    case SOP_F32: e = adjoint_k<SOP_F32>(k, s); break;
    case SOP_BF16: e = adjoint_k<SOP_BF16>(k, s); break;
    case SOP_F16: e = adjoint_k<SOP_F16>(k, s); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    const int64_t ne = (int64_t)a.He * a.We;
    env_fold_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, s>>>(k.genv4, ne, a.g_env);
    return cudaGetLastError();
}

}  // namespace sop
