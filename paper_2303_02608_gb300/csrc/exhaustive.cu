// Regression pass 1 of exhaustive frames: every pixel, window sums factored over
// the frames.
//
// At a window offset the frames are summed first (accp_neighbour), then the
// coordinates are multiplied in (accp_offset), which needs all frames of the
// window at once: a tile of 16 x 4 pixels plus halo of as many frames as fit
// half an SM's shared memory is staged together by TMA (more frames come in
// equal groups).  Four lanes share a pixel, lane l taking offsets l, l + 4, ...,
// which keeps the tile small, lets small images fill the chip (a tile of one
// lane per pixel leaves 333 x 251 pixels with one wave and a sixth) and cuts
// a pixel's sums into four shorter ones.  The division is the same for every
// image size: a pixel's sums are rounded the same way in any image or strip.
// Of a warp's lanes each quarter reads 8 neighbouring records: no bank
// conflicts.  Offsets outside the image get weight 0 through their distance
// (the copy fills them with zeros).  While a tile's sums are reduced and stored
// the next tile's first group lands; the other CTA of the SM covers the rest.
//
// FP32-bound, 70% of the FMA pipe.  1920 x 1080, 15 x 15 x 5 window, precision
// form: 6.92 ms, against 7.36 ms for the tile-staged kernel (7.17 without
// unrolling the frames by two, 7.74 with the first frame peeled); 333 x 251,
// 11 x 11 x 4, FP32: 154 us against 189.  Its alpha is also nearer to float64
// (3e-7 against 2e-6, relative).
//
// Frame 0 of an adaptive sequence stays with the tile-staged kernel: its sums
// decide where that sequence's events fall, and rounding them in another order
// would move a few events of every sequence.
#include "internal.h"
#include "ptx.cuh"
#include "wlr_math.cuh"

namespace esim {
namespace {

struct ExhaustiveLayout {
    int frame, group, table, total;   // bytes per staged frame, frames staged together, table offset, all bytes
};

__host__ __device__ inline ExhaustiveLayout exhaustive_layout(int r, int T, bool mixed, int budget)
{
    ExhaustiveLayout L;
    const int tw = kExTileX + 2 * r, th = kExTileY + 2 * r, nq = (2 * r + 1) * (2 * r + 1);
    L.frame = ((mixed ? 1 : 2) * tw * th * 16 + 127) & ~127;
    const int fixed = nq * 16 + 128;
    int fit = (budget - fixed) / L.frame;
    fit = fit < 1 ? 1 : fit > T ? T : fit;
    const int groups = (T + fit - 1) / fit;
    L.group = (T + groups - 1) / groups;
    L.table = L.group * L.frame;
    L.total = L.table + fixed;
    return L;
}

template <bool kMixed>
__global__ void __launch_bounds__(kTilePix, 2)
    exhaustive_kernel(const __grid_constant__ CUtensorMap tmap, const WlrParams p)
{
    constexpr int kLanes = kExLanes, kTH = kExTileY, kWarpPix = 32 / kLanes, kAcross = kExTileX / kWarpPix;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
    __shared__ uint64_t full;
    __shared__ int s_next[2];
    __shared__ unsigned long long s_pairs, s_pix;
    const int side = 2 * p.r + 1, nq = side * side;
    const int sw = kExTileX + 2 * p.r, plane = sw * (kTH + 2 * p.r);
    const int frame_bytes = ((kMixed ? 1 : 2) * plane * 16 + 127) & ~127;
    const int tiles_x = (p.W + kExTileX - 1) / kExTileX;
    const int n_items = tiles_x * ((p.H + kTH - 1) / kTH);
    const float spx = p.s_coord_px;
    // (u_dx, u_dy, -(u_dx^2 + u_dy^2), record offset | (dx + 16) << 16 | (dy + 16) << 24)
    float4* table = reinterpret_cast<float4*>(smem + p.frame_group * frame_bytes);
    for (int q = threadIdx.x; q < nq; q += kTilePix) {
        const int ox = q % side - p.r, oy = q / side - p.r;
        const float u1 = (float)ox * spx, u2 = (float)oy * spx;
        table[q] = make_float4(u1, u2, -fmaf(u1, u1, u2 * u2),
                               __int_as_float(((oy * sw + ox) & 0xffff) | (ox + 16) << 16 | (oy + 16) << 24));
    }
    auto issue = [&](int item, int k0) {
        const int tx0 = (item % tiles_x) * kExTileX, ty0 = (item / tiles_x) * kTH;
        const int n = min(p.frame_group, p.n_tau - k0);
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&full, (uint32_t)(n * (kMixed ? 1 : 2) * plane * 16));
        for (int k = 0; k < n; ++k) {
            const int slot = (p.t - k0 - k) % p.T;
            tma_load_4d(smem + k * frame_bytes, &tmap, &full, 0, tx0 - p.r, ty0 - p.r, kMixed ? slot : 2 * slot);
        }
    };
    if (threadIdx.x == 0) {
        mbar_init(&full, 1);
        mbar_fence_init();
        s_pairs = 0ull;
        s_pix = 0ull;
        s_next[1] = (int)atomicAdd(&p.ctrl->work_next, 1u);
        if (s_next[1] < n_items) issue(s_next[1], 0);
    }
    __syncthreads();
    int item = s_next[1], par = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane / kWarpPix;
    const int lx = (warp % kAcross) * kWarpPix + lane % kWarpPix, ly = warp / kAcross;
    const int centre = (ly + p.r) * sw + lx + p.r;
    const float* sf = kMixed ? p.q_scale : p.s_feat;   // regressor scale of a stored value
    AccP acc;
    PairConst kc;
    uint32_t phase = 0u;
    bool timed_out = false;
    while (item < n_items) {
        const int tx0 = (item % tiles_x) * kExTileX, ty0 = (item / tiles_x) * kTH;
        const int cx = tx0 + lx, cy = ty0 + ly;
        const bool interior = tx0 >= p.r && ty0 >= p.r && tx0 + kExTileX + p.r <= p.W && ty0 + kTH + p.r <= p.H;
        accp_zero(acc);
        int next = 0;
        for (int k0 = 0; k0 < p.n_tau; k0 += p.frame_group) {
            const int n = min(p.frame_group, p.n_tau - k0);
            const bool ok = mbar_wait_bounded(&full, phase);
            phase ^= 1u;
            if (k0 == 0 && threadIdx.x == 0) s_next[par] = (int)atomicAdd(&p.ctrl->work_next, 1u);
            if (ok) {
                const uint4* PM = reinterpret_cast<const uint4*>(smem);
                const float4* PF = reinterpret_cast<const float4*>(smem);
                const int fstep = frame_bytes / 16;
                if (k0 == 0) {   // the first staged frame is t: the centre's features
                    float c[7];
                    if (kMixed) {
                        float yc;
                        unpack_mixed(PM[centre], yc, c);
                    } else {
                        const float4 c0 = PF[centre], c1 = PF[plane + centre];
                        c[0] = c0.y; c[1] = c0.z; c[2] = c0.w; c[3] = c1.x; c[4] = c1.y; c[5] = c1.z; c[6] = c1.w;
                    }
                    float cf[7];
#pragma unroll
                    for (int j = 0; j < 7; ++j) cf[j] = c[j] * sf[j];
                    kc = pair_const(sf, cf);
                }
#pragma unroll 1
                for (int q = sub; q < nq; q += kLanes) {
                    const float4 e = table[q];
                    const int bits = __float_as_int(e.w);
                    float en0 = e.z;
                    if (!interior) {
                        const int x = cx + ((bits >> 16) & 0xff) - 16, y = cy + ((bits >> 24) & 0xff) - 16;
                        if (x < 0 || x >= p.W || y < 0 || y >= p.H) en0 = -1e30f;
                    }
                    int at = centre + (int)(short)bits;
                    OffSums o;
                    offsums_zero(o);
#pragma unroll 2
                    for (int k = 0; k < n; ++k) {
                        if (kMixed) accp_neighbour(acc, o, en0, PM[at], kc);
                        else accp_neighbour(acc, o, en0, PF[at], PF[at + plane], kc);
                        at += fstep;
                    }
                    accp_offset(acc, o, make_float2(e.x, e.y));
                }
            }
            if (__syncthreads_or(!ok)) {   // every warp is past its reads of the staged frames
                timed_out = true;
                break;
            }
            next = s_next[par];
            if (threadIdx.x == 0) {
                if (k0 + p.frame_group < p.n_tau) issue(item, k0 + p.frame_group);
                else if (next < n_items) issue(next, 0);
            }
        }
        if (timed_out) break;
        accp_reduce<32 / kLanes>(acc, kLanes);
        if (cx < p.W && cy < p.H) {
            accp_store(acc, p.gram + ((size_t)cy * p.W + cx) * kGramStride, sub, kLanes);
            if (sub == 0) {
                const int nx = min(p.W - 1, cx + p.r) - max(0, cx - p.r) + 1;
                const int ny = min(p.H - 1, cy + p.r) - max(0, cy - p.r) + 1;
                atomicAdd(&s_pairs, (unsigned long long)(nx * ny * p.n_tau));
                atomicAdd(&s_pix, 1ull);
            }
        }
        item = next;
        par ^= 1;   // a slow warp may still read the other slot
    }
    // a copy that did not land in time gets one more bounded wait before the CTA exits
    if (timed_out) mbar_wait_bounded(&full, phase ^ 1u, 1u << 20);
    __syncthreads();
    finish(p, s_pairs, s_pix, 0ull, timed_out, false);
}

}  // namespace

int exhaustive_smem(int r, int T, bool mixed, int max_smem_per_sm, int* group)
{
    const int budget = max_smem_per_sm / 2 - 1024 - 256;   // two CTAs per SM; the system's 1 KB, static variables
    const ExhaustiveLayout L = exhaustive_layout(r, T, mixed, budget);
    *group = L.group;
    return L.total;
}

cudaError_t exhaustive_prepare(int max_smem_block, bool mixed)
{
    // the device's limit, not this context's need: contexts of other radii launch the same kernel
    const void* k = mixed ? (const void*)exhaustive_kernel<true> : (const void*)exhaustive_kernel<false>;
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, k);
    return e != cudaSuccess ? e
                            : cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   max_smem_block - (int)a.sharedSizeBytes);
}

int exhaustive_grid(int smem_bytes, int num_sms, int W, int H, bool mixed)
{
    int per_sm = 0;
    const cudaError_t e =
        mixed ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, exhaustive_kernel<true>, kTilePix, smem_bytes)
              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, exhaustive_kernel<false>, kTilePix, smem_bytes);
    if (e != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const int tiles = ((W + kExTileX - 1) / kExTileX) * ((H + kExTileY - 1) / kExTileY);
    return tiles < per_sm * num_sms ? tiles : per_sm * num_sms;
}

cudaError_t launch_exhaustive(const CUtensorMap& tmap, const WlrParams& p, bool mixed, int grid, int smem_bytes,
                              cudaStream_t s)
{
    if (mixed)
        exhaustive_kernel<true><<<grid, kTilePix, smem_bytes, s>>>(tmap, p);
    else
        exhaustive_kernel<false><<<grid, kTilePix, smem_bytes, s>>>(tmap, p);
    return cudaGetLastError();
}

}  // namespace esim
