// Regression pass 1 of exhaustive frames: every pixel, window sums factored over
// the frames.
//
// At a window offset the frames are summed first (accp_neighbour), then the
// coordinates are multiplied in (accp_offset), which needs all frames of the
// window at once: a tile of 16 x 4 pixels plus halo of every frame is staged
// together by TMA, in at most half an SM's shared memory.  Four lanes share a
// pixel, lane l taking offsets l, l + 4, ..., which keeps the tile small, lets
// small images fill the chip and cuts a pixel's sums into four shorter ones.
// Of a warp's lanes each quarter reads 8 neighbouring records: no bank
// conflicts.  Offsets outside the image get weight 0 through their distance
// (the copy fills them with zeros); those outside for every pixel are left out
// (a frame of 17 x 5, 21 x 21 x 4 window: 107 us, 130 with them, 125 tile-staged).
// While a tile's sums are reduced and stored the next tile's frames land; the
// other CTA of the SM covers the rest.
//
// It takes the windows where it wins at the image sizes measured: radius 7 and up, at
// least 4 frames (5 in the FP32 form, whose records cost no unpacking that the
// factored sums could share), and all frames of a tile fitting together.  Fewer
// frames or offsets do not repay the work per offset and the four lanes' sum.
// A frame of 1500 x 1000 / 200 x 150 in microseconds, tile-staged -> here:
// precision form, radius 7, 5 frames 5561 / 228 -> 5320 / 197; 4 frames 4498 / 199
// -> 4494 / 174; FP32, 5 frames 5216 / 219 -> 5152 / 197.  Not taken: FP32, 4 frames
// 4215 / 191 -> 4415 / 174; radius 5, 4 frames, precision form 2567 / 141 -> 2612 /
// 122; with frames in two groups (FP32, radius 9, 5 frames) 900 x 700 3613 -> 4109.
// Whole frames of the other windows that fit, tile-staged / here, 16 windows
// (precision form: radius 7 with 4 to 12 frames, 8 and 9 with 4 and 5, 10 to 13 with 4;
// FP32: radius 7 with 5 and 6, 8 with 5): 1500 x 1000 1.01-1.13, 640 x 480 1.01-1.16, 333 x 251
// 1.28-1.47, 200 x 150 1.07-1.21, 64 x 48 2.0-2.9.  Only images of a few pixels lose, by
// the window's part that reaches no pixel: 5 x 17, 27 x 27 x 4 window 132 us for 124.
// The choice does not look at the image's size: a pixel's sums are rounded the
// same way in any image or strip.
//
// FP32-bound: the FMA pipe is 70% busy (960 x 540).  1920 x 1080, 15 x 15 x 5 window, precision
// form: a frame takes 7.32 ms, 7.65 with the tile-staged kernel (the frames'
// loop not unrolled costs 3% more, its first frame peeled 8%).  Its alpha is also
// nearer to float64 (3e-7 against 2e-6, relative).
//
// Frame 0 of an adaptive sequence stays with the tile-staged kernel: its sums
// decide where that sequence's events fall, and rounding them in another order
// would move a few events of every sequence.
#include "internal.h"
#include "ptx.cuh"
#include "wlr_math.cuh"

namespace esim {
namespace {

// Bytes of a staged frame.
__host__ __device__ inline int frame_bytes(int r, bool mixed)
{
    return ((mixed ? 1 : 2) * (kExTileX + 2 * r) * (kExTileY + 2 * r) * 16 + 127) & ~127;
}

// Add a pixel's four lanes (8 apart) and store its record.  Every lane needs
// only the quarter of the 17 quads that it stores (quad q by lane q % 4), so
// each step passes on the half that the other side keeps: 52 shuffles, where
// adding everything in every lane takes 132 (6% of an 11 x 11 x 4 window's
// time).  Same tree, same bits.
__device__ __forceinline__ void fold_store(const AccP& a, float* __restrict__ rec, int sub, bool live)
{
    static_assert(kExLanes == 4 && kGramStride == 68, "two halvings of 16 quads, and one quad more");
    float v[kGramStride];
    accp_values(a, v);
    const bool b1 = sub & 2, b0 = sub & 1;
    float m[32], o[16];
#pragma unroll
    for (int i = 0; i < 32; ++i) {   // quads 4j, 4j + 1 of lanes 0, 1; 4j + 2, 4j + 3 of lanes 2, 3
        const int lo = (i >> 3) * 16 + (i & 7), hi = lo + 8;
        m[i] = (b1 ? v[hi] : v[lo]) + __shfl_xor_sync(0xffffffffu, b1 ? v[lo] : v[hi], 16);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int lo = (i >> 2) * 8 + (i & 3), hi = lo + 4;
        o[i] = (b0 ? m[hi] : m[lo]) + __shfl_xor_sync(0xffffffffu, b0 ? m[lo] : m[hi], 8);
    }
    float t[2];   // quad 16: its last two are padding
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        t[i] = v[64 + i] + __shfl_xor_sync(0xffffffffu, v[64 + i], 16);
        t[i] += __shfl_xor_sync(0xffffffffu, t[i], 8);
    }
    if (!live) return;
    float4* out = reinterpret_cast<float4*>(rec);
#pragma unroll
    for (int j = 0; j < 4; ++j) out[4 * j + sub] = make_float4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
    if (sub == 0) out[16] = make_float4(t[0], t[1], 0.0f, 0.0f);
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
    const int fbytes = frame_bytes(p.r, kMixed);
    const int tiles_x = (p.W + kExTileX - 1) / kExTileX;
    const int n_items = tiles_x * ((p.H + kTH - 1) / kTH);
    const float spx = p.s_coord_px;
    // (u_dx, u_dy, -(u_dx^2 + u_dy^2), record offset | (dx + 16) << 16 | (dy + 16) << 24)
    float4* table = reinterpret_cast<float4*>(smem + p.T * fbytes);
    const int rx = min(p.r, p.W - 1), ry = min(p.r, p.H - 1);   // offsets beyond these reach no pixel of the image
    const bool whole = rx == p.r && ry == p.r;
    __shared__ int s_steps;   // entries per lane
    if (threadIdx.x == 0) s_steps = whole ? (nq + kLanes - 1) / kLanes : 0;
    if (!whole) {
        const float4 none = make_float4(0.0f, 0.0f, -1e30f, __int_as_float(16 << 16 | 16 << 24));
        for (int q = threadIdx.x; q < nq; q += kTilePix) table[q] = none;
        __syncthreads();
    }
    for (int q = threadIdx.x; q < nq; q += kTilePix) {
        const int ox = q % side - p.r, oy = q / side - p.r;
        const float u1 = (float)ox * spx, u2 = (float)oy * spx;
        int at = q;
        if (!whole) {
            // in an image smaller than the window each lane's list closes up over the others (entries
            // of weight 0 even out the lists), so that every lane adds the same offsets in the same order
            if (abs(ox) > rx || abs(oy) > ry) continue;
            at = q % kLanes;
            for (int k = q % kLanes; k < q; k += kLanes)
                if (abs(k % side - p.r) <= rx && abs(k / side - p.r) <= ry) at += kLanes;
            atomicMax(&s_steps, at / kLanes + 1);
        }
        table[at] = make_float4(u1, u2, -fmaf(u1, u1, u2 * u2),
                                __int_as_float(((oy * sw + ox) & 0xffff) | (ox + 16) << 16 | (oy + 16) << 24));
    }
    auto issue = [&](int item) {
        const int tx0 = (item % tiles_x) * kExTileX, ty0 = (item / tiles_x) * kTH;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&full, (uint32_t)(p.n_tau * (kMixed ? 1 : 2) * plane * 16));
        for (int k = 0; k < p.n_tau; ++k) {
            const int slot = (p.t - k) % p.T;
            tma_load_4d(smem + k * fbytes, &tmap, &full, 0, tx0 - p.r, ty0 - p.r, kMixed ? slot : 2 * slot);
        }
    };
    if (threadIdx.x == 0) {
        mbar_init(&full, 1);
        mbar_fence_init();
        s_pairs = 0ull;
        s_pix = 0ull;
        s_next[1] = (int)atomicAdd(&p.ctrl->work_next, 1u);
        if (s_next[1] < n_items && !p.withhold_copy) issue(s_next[1]);   // withheld (test): the phase never completes
    }
    __syncthreads();
    int item = s_next[1], par = 0;
    const int n_off = min(nq, kLanes * s_steps);
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
        const bool ok = mbar_wait_bounded(&full, phase, p.poll_limit);
        phase ^= 1u;
        if (threadIdx.x == 0) s_next[par] = (int)atomicAdd(&p.ctrl->work_next, 1u);
        if (ok) {
            const uint4* PM = reinterpret_cast<const uint4*>(smem);
            const float4* PF = reinterpret_cast<const float4*>(smem);
            const int fstep = fbytes / 16;
            {   // the first staged frame is t: the centre's features
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
            for (int q = sub; q < n_off; q += kLanes) {
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
                for (int k = 0; k < p.n_tau; ++k) {
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
        const int next = s_next[par];
        if (threadIdx.x == 0 && next < n_items) issue(next);
        const bool live = cx < p.W && cy < p.H;
        fold_store(acc, p.gram + ((size_t)cy * p.W + cx) * kGramStride, sub, live);
        if (live) {
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
    if (timed_out) mbar_wait_bounded(&full, phase ^ 1u, p.poll_limit);
    __syncthreads();
    finish(p, s_pairs, s_pix, 0ull, timed_out, false);
}

}  // namespace

int exhaustive_smem(int r, int T, bool mixed, int max_smem_per_sm)
{
    const int budget = max_smem_per_sm / 2 - 1024 - 256;   // two CTAs per SM; the system's 1 KB, static variables
    const int total = T * frame_bytes(r, mixed) + (2 * r + 1) * (2 * r + 1) * 16 + 128;   // + alignment slack
    return r >= 7 && T >= (mixed ? 4 : 5) && total <= budget ? total : 0;
}

cudaError_t exhaustive_prepare(int max_smem_block, bool mixed)
{
    return allow_dynamic_smem(mixed ? (const void*)exhaustive_kernel<true> : (const void*)exhaustive_kernel<false>,
                              max_smem_block);
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
