// Monte Carlo renderer for analytic test scenes: produces the simulator's
// inputs (noisy radiance, variance of the luminance estimate, first-hit
// normal, depth and albedo) for an open-fronted room with an area light and
// moving spheres.  Every floating-point operation is an explicitly rounded
// IEEE FP32 operation (no fused multiply-add contraction), so each pixel is a
// fixed function of scene, frame and seed that a plain FP32 restatement can
// reproduce bit for bit.
//
// One thread per pixel; samples in order; per sample a jittered camera ray
// and up to max_bounces surface interactions, each with next-event estimation
// towards one uniform point of the light and a cosine-weighted bounce.  The
// kernel is bound by instruction issue (83% of the slots): one kernel per
// number of spheres, so that their loops unroll; what depends on the scene
// alone is formed once per block; a ray's walls take one division per axis
// whatever its signs; the offsets from a hit point to the spheres serve both
// its shadow ray and the bounce that leaves it; a shadow ray stops at its first
// blocker.  All of it with the same operations on the same values.  1920 x 1080,
// 4 samples, two interactions: 301 us with three spheres (336 before), 224 / 244
// with none, 457 / 523 with eight.  Keeping the spheres' offsets takes
// registers: four CTAs per SM up to four spheres, three beyond, measured faster
// than what the compiler chooses (354 us at two per SM).
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), key
// (seed, frame), counter (pixel, sample, call, 0); call 1 gives the pixel
// jitter, call 2b + 2 the light point and bounce direction of interaction b.
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace esim {
namespace {

// explicitly rounded FP32 arithmetic
__device__ __forceinline__ float fa(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fs(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fm(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fd(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fq(float a) { return __fsqrt_rn(a); }

struct V3 {
    float x, y, z;
};
__device__ __forceinline__ V3 v3(float x, float y, float z) { return V3{x, y, z}; }
__device__ __forceinline__ V3 vsub(V3 a, V3 b) { return v3(fs(a.x, b.x), fs(a.y, b.y), fs(a.z, b.z)); }
__device__ __forceinline__ V3 vscale(V3 a, float s) { return v3(fm(a.x, s), fm(a.y, s), fm(a.z, s)); }
__device__ __forceinline__ float vdot(V3 a, V3 b) { return fa(fa(fm(a.x, b.x), fm(a.y, b.y)), fm(a.z, b.z)); }
// o + t d
__device__ __forceinline__ V3 vray(V3 o, float t, V3 d) { return v3(fa(o.x, fm(t, d.x)), fa(o.y, fm(t, d.y)), fa(o.z, fm(t, d.z))); }

// Philox4x32-10 bijection of a 128-bit counter under a 64-bit key.
__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
        const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

// uniform in [0, 1): the top 24 bits of a word, exactly representable
__device__ __forceinline__ float unit(uint32_t w) { return fm((float)(w >> 8), 5.9604644775390625e-8f); }

// cos and sin of 2 pi u, u in [0, 1): quarter-turn reduction, then the
// Taylor polynomials of sin and cos on [0, pi/2) (truncation below 1e-7).
__device__ __forceinline__ void sincos_turns(float u, float& c, float& s)
{
    const float u4 = fm(u, 4.0f);
    const float qf = floorf(u4);
    const int q = (int)qf;
    const float th = fm(fs(u4, qf), 1.57079637f);
    const float t2 = fm(th, th);
    float ps = -2.50521084e-8f;   // -1/11!
    ps = fa(fm(ps, t2), 2.75573188e-6f);
    ps = fa(fm(ps, t2), -1.98412701e-4f);
    ps = fa(fm(ps, t2), 8.33333377e-3f);
    ps = fa(fm(ps, t2), -1.66666672e-1f);
    ps = fa(fm(ps, t2), 1.0f);
    const float sn = fm(ps, th);
    float pc = 2.08767570e-9f;    // 1/12!
    pc = fa(fm(pc, t2), -2.75573188e-7f);
    pc = fa(fm(pc, t2), 2.48015876e-5f);
    pc = fa(fm(pc, t2), -1.38888892e-3f);
    pc = fa(fm(pc, t2), 4.16666679e-2f);
    pc = fa(fm(pc, t2), -0.5f);
    const float cs = fa(fm(pc, t2), 1.0f);
    if (q == 0) { c = cs; s = sn; }
    else if (q == 1) { c = -sn; s = cs; }
    else if (q == 2) { c = -cs; s = -sn; }
    else { c = sn; s = -cs; }
}

struct Hit {
    float t;
    int kind;   // 0..4 walls (left, right, floor, ceiling, back), 5 open front, 8 + j sphere j
};

// What a block forms once from the scene and the frame.
template <int N>
struct Tables {
    float4 surf[16][2];       // by hit kind: albedo and, for spheres, 1 / radius; normal or sphere centre
    float4 cam[N ? N : 1];    // camera - centre and |.|^2 - radius^2
    float4 ctr[N ? N : 1];    // centre, radius^2
};

// |oc|^2 - r^2 of a ray's origin seen from a sphere (oc = origin - centre).
__device__ __forceinline__ float4 from_sphere(V3 o, float4 c)
{
    const V3 oc = vsub(o, v3(c.x, c.y, c.z));
    return make_float4(oc.x, oc.y, oc.z, fs(vdot(oc, oc), c.w));
}

// Distance to the nearer intersection beyond eps, or a value not above eps.
__device__ __forceinline__ float hit_sphere(float4 oc, V3 d, float eps)
{
    const float b = vdot(v3(oc.x, oc.y, oc.z), d);
    const float disc = fs(fm(b, b), oc.w);
    if (!(disc > 0.0f)) return 0.0f;
    const float sq = fq(disc);
    const float t = fs(-b, sq);
    return t > eps ? t : fa(-b, sq);
}

// The wall (or the open front) a ray from inside the room reaches; a direction
// that is not a number reaches none.
__device__ __forceinline__ Hit hit_walls(const esim_ad_render_scene& sc, V3 o, V3 d)
{
    Hit h{INFINITY, 5};
    const float tx = fd(fs(d.x > 0.0f ? sc.box[0] : -sc.box[0], o.x), d.x);
    if (fabsf(d.x) > 0.0f) {
        h.t = tx;
        h.kind = d.x > 0.0f ? 1 : 0;
    }
    const float ty = fd(fs(d.y > 0.0f ? sc.box[1] : -sc.box[1], o.y), d.y);
    if (fabsf(d.y) > 0.0f && ty < h.t) {
        h.t = ty;
        h.kind = d.y > 0.0f ? 3 : 2;
    }
    const float tz = fd(fs(d.z > 0.0f ? sc.box[2] : -sc.box[2], o.z), d.z);
    if (fabsf(d.z) > 0.0f && tz < h.t) {
        h.t = tz;
        h.kind = d.z > 0.0f ? 5 : 4;
    }
    return h;
}

template <int N>
__global__ void __launch_bounds__(256, N <= 4 ? 4 : 3) render_kernel(const esim_ad_render_scene sc, int frame,
                                                     float* __restrict__ radiance, float* __restrict__ variance,
                                                     float* __restrict__ normal, float* __restrict__ albedo,
                                                     float* __restrict__ depth)
{
    __shared__ Tables<N> tab;
    const V3 cam = v3(sc.cam_pos[0], sc.cam_pos[1], sc.cam_pos[2]);
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    if (tid < 5) {
        const float nx = tid == 0 ? 1.0f : tid == 1 ? -1.0f : 0.0f, ny = tid == 2 ? 1.0f : tid == 3 ? -1.0f : 0.0f;
        tab.surf[tid][0] = make_float4(sc.wall_albedo[tid][0], sc.wall_albedo[tid][1], sc.wall_albedo[tid][2], 0.0f);
        tab.surf[tid][1] = make_float4(nx, ny, tid == 4 ? 1.0f : 0.0f, 0.0f);
    }
    if (tid >= 32 && tid < 32 + N) {
        const int j = tid - 32;
        const esim_ad_sphere& sp = sc.spheres[j];
        const float tf = (float)frame;
        const float4 c = make_float4(fa(sp.center[0], fm(tf, sp.velocity[0])), fa(sp.center[1], fm(tf, sp.velocity[1])),
                                     fa(sp.center[2], fm(tf, sp.velocity[2])), fm(sp.radius, sp.radius));
        tab.ctr[j] = c;
        tab.cam[j] = from_sphere(cam, c);
        tab.surf[8 + j][0] = make_float4(sp.albedo[0], sp.albedo[1], sp.albedo[2], fd(1.0f, sp.radius));
        tab.surf[8 + j][1] = c;
    }
    __syncthreads();
    const int px = blockIdx.x * blockDim.x + threadIdx.x;
    const int py = blockIdx.y * blockDim.y + threadIdx.y;
    if (px >= sc.width || py >= sc.height) return;
    const size_t NP = (size_t)sc.width * sc.height;
    const uint32_t pix = (uint32_t)py * (uint32_t)sc.width + (uint32_t)px;
    const float tany = sc.tan_half_fov_y;
    const float tanx = fd(fm(tany, (float)sc.width), (float)sc.height);
    const float lw = fs(sc.light[1], sc.light[0]), lh = fs(sc.light[3], sc.light[2]);
    const float area = fm(lw, lh);
    float sum[3] = {0.0f, 0.0f, 0.0f}, sy = 0.0f, sy2 = 0.0f;
    float fn[3] = {0.0f, 0.0f, 0.0f}, fal[3] = {0.0f, 0.0f, 0.0f}, fdp = 0.0f;
    for (int smp = 0; smp < sc.spp; ++smp) {
        const uint4 jit = philox(pix, (uint32_t)smp, 1u, 0u, sc.seed, (uint32_t)frame);
        const float sxp = fm(fs(fm(fd(fa((float)px, unit(jit.x)), (float)sc.width), 2.0f), 1.0f), tanx);
        const float syp = fm(fs(1.0f, fm(fd(fa((float)py, unit(jit.y)), (float)sc.height), 2.0f)), tany);
        const float inv = fd(1.0f, fq(fa(fa(fm(sxp, sxp), fm(syp, syp)), 1.0f)));
        V3 o = cam;
        V3 d = v3(fm(sxp, inv), fm(syp, inv), -inv);
        float4 oc[N ? N : 1];   // the ray's origin from the spheres
#pragma unroll
        for (int j = 0; j < N; ++j) oc[j] = tab.cam[j];
        float thr[3] = {1.0f, 1.0f, 1.0f};
        float L[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 1
        for (int b = 0; b < sc.max_bounces; ++b) {
            Hit h = hit_walls(sc, o, d);
            Hit hs{INFINITY, -1};
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const float t = hit_sphere(oc[j], d, sc.eps);
                if (t > sc.eps && t < hs.t) {
                    hs.t = t;
                    hs.kind = 8 + j;
                }
            }
            if (hs.t < h.t) h = hs;
            if (h.kind == 5) break;   // out through the open front
            const V3 x = vray(o, h.t, d);
            const float4 e0 = tab.surf[h.kind][0], e1 = tab.surf[h.kind][1];
            float al[3] = {e0.x, e0.y, e0.z};
            V3 n = v3(e1.x, e1.y, e1.z);
            if (h.kind >= 8) {
                n = vscale(vsub(x, n), e0.w);
            } else if (h.kind == 4 && sc.checker > 0.0f) {
                const float ix = floorf(fd(x.x, sc.checker)), iy = floorf(fd(x.y, sc.checker));
                if (((int)ix + (int)iy) & 1)
                    for (int c = 0; c < 3; ++c) al[c] = sc.back_albedo2[c];
            }
            if (b == 0) {
                fn[0] = fa(fn[0], n.x);
                fn[1] = fa(fn[1], n.y);
                fn[2] = fa(fn[2], n.z);
                for (int c = 0; c < 3; ++c) fal[c] = fa(fal[c], al[c]);
                fdp = fa(fdp, h.t);
            }
            if (h.kind == 3 && x.x >= sc.light[0] && x.x <= sc.light[1] && x.z >= sc.light[2] && x.z <= sc.light[3]) {
                if (b == 0)   // emission, seen by camera rays only
                    for (int c = 0; c < 3; ++c) L[c] = fa(L[c], sc.light_radiance[c]);
                break;
            }
#pragma unroll
            for (int j = 0; j < N; ++j) oc[j] = from_sphere(x, tab.ctr[j]);
            const uint4 r = philox(pix, (uint32_t)smp, (uint32_t)(2 * b + 2), 0u, sc.seed, (uint32_t)frame);
            // next-event estimation: one uniform point of the light
            const V3 lp = v3(fa(sc.light[0], fm(unit(r.x), lw)), sc.box[1], fa(sc.light[2], fm(unit(r.y), lh)));
            const V3 w = vsub(lp, x);
            const float d2 = vdot(w, w);
            const float dist = fq(d2);
            const V3 wl = vscale(w, fd(1.0f, dist));
            const float cs = vdot(n, wl);
            const float cl = wl.y;
            if (cs > 0.0f && cl > 0.0f) {
                const float lim = fs(dist, sc.eps);
                bool blocked = false;
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    if (blocked) break;
                    const float t = hit_sphere(oc[j], wl, sc.eps);
                    blocked = t > sc.eps && t < lim;
                }
                if (!blocked) {
                    const float g = fd(fm(fm(cs, cl), area), fm(3.14159274f, d2));
                    for (int c = 0; c < 3; ++c)
                        L[c] = fa(L[c], fm(fm(fm(thr[c], al[c]), sc.light_radiance[c]), g));
                }
            }
            if (b + 1 >= sc.max_bounces) break;
            // cosine-weighted bounce around n (basis of Duff et al. 2017)
            float cph, sph;
            sincos_turns(unit(r.w), cph, sph);
            const float rr = fq(unit(r.z));
            const float lz = fq(fmaxf(fs(1.0f, unit(r.z)), 0.0f));
            const float lx = fm(rr, cph), ly = fm(rr, sph);
            const float sg = n.z >= 0.0f ? 1.0f : -1.0f;
            const float aa = fd(-1.0f, fa(sg, n.z));
            const float bb = fm(fm(n.x, n.y), aa);
            const V3 t1 = v3(fa(1.0f, fm(fm(sg, fm(n.x, n.x)), aa)), fm(sg, bb), -fm(sg, n.x));
            const V3 t2 = v3(bb, fa(sg, fm(fm(n.y, n.y), aa)), -n.y);
            d = v3(fa(fa(fm(t1.x, lx), fm(t2.x, ly)), fm(n.x, lz)),
                   fa(fa(fm(t1.y, lx), fm(t2.y, ly)), fm(n.y, lz)),
                   fa(fa(fm(t1.z, lx), fm(t2.z, ly)), fm(n.z, lz)));
            o = x;
            for (int c = 0; c < 3; ++c) thr[c] = fm(thr[c], al[c]);
        }
        for (int c = 0; c < 3; ++c) sum[c] = fa(sum[c], L[c]);
        const float Y = fa(fa(fm(0.2126f, L[0]), fm(0.7152f, L[1])), fm(0.0722f, L[2]));
        sy = fa(sy, Y);
        sy2 = fa(sy2, fm(Y, Y));
    }
    const float n = (float)sc.spp;
    for (int c = 0; c < 3; ++c) {
        radiance[c * NP + pix] = fd(sum[c], n);
        normal[c * NP + pix] = fd(fn[c], n);
        albedo[c * NP + pix] = fd(fal[c], n);
    }
    depth[pix] = fd(fdp, n);
    float v = 0.0f;
    if (sc.spp > 1) v = fmaxf(fd(fs(sy2, fd(fm(sy, sy), n)), fm(n, fs(n, 1.0f))), 0.0f);
    variance[pix] = v;
}

typedef void (*RenderKernel)(const esim_ad_render_scene, int, float*, float*, float*, float*, float*);
const RenderKernel kRender[9] = {render_kernel<0>, render_kernel<1>, render_kernel<2>, render_kernel<3>, render_kernel<4>,
                                 render_kernel<5>, render_kernel<6>, render_kernel<7>, render_kernel<8>};

}  // namespace
}  // namespace esim

using namespace esim;

extern "C" esim_ad_status esim_ad_render(const esim_ad_render_scene* scene, int32_t frame, float* radiance,
                                         float* variance, float* normal, float* albedo, float* depth,
                                         void* cuda_stream)
{
    if (!scene || !radiance || !variance || !normal || !albedo || !depth) return ESIM_AD_EINVAL;
    const esim_ad_render_scene& s = *scene;
    if (s.struct_size != sizeof(esim_ad_render_scene) || s.width < 1 || s.height < 1 ||
        (long long)s.width * s.height >= (1ll << 31) || s.spp < 1 || s.spp > 65536 || s.max_bounces < 1 ||
        s.max_bounces > 8 || s.n_spheres < 0 || s.n_spheres > 8 || !(s.tan_half_fov_y > 0.0f) ||
        !(s.box[0] > 0.0f) || !(s.box[1] > 0.0f) || !(s.box[2] > 0.0f) || !(s.light[1] > s.light[0]) ||
        !(s.light[3] > s.light[2]) || !(s.eps > 0.0f) || frame < 0)
        return ESIM_AD_EINVAL;
    for (int j = 0; j < s.n_spheres; ++j)
        if (!(s.spheres[j].radius > 0.0f)) return ESIM_AD_EINVAL;
    const dim3 block(16, 16);
    const dim3 grid((s.width + 15) / 16, (s.height + 15) / 16);
    kRender[s.n_spheres]<<<grid, block, 0, (cudaStream_t)cuda_stream>>>(s, frame, radiance, variance, normal, albedo,
                                                                       depth);
    return cudaGetLastError() == cudaSuccess ? ESIM_AD_OK : ESIM_AD_ECUDA;
}
