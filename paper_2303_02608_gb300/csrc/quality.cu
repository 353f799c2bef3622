// Evaluation kernels (Section 3, quantitative comparison): the plain ESIM
// simulator, and polarity-aware precision, recall, F-score and chamfer
// distance between two event sets with an exact nearest-neighbour search.
//
// Events are signed points (x / W, y / H, t / F).  For one set and each
// polarity, a column pass stores per pixel and frame the distance in rows to
// the nearest event of that polarity in the pixel's column (g).  The nearest
// event of a query (x, y, t) is then
//     min over t', q of ((x - q) / W)^2 + (g_t'(q, y) / H)^2 + ((t - t') / F)^2,
// searched outward in |t - t'| and |x - q| and cut off as soon as the
// separation alone reaches the best squared distance found.  Frames without
// any event of the polarity are skipped through a per-frame flag.  Sums of the
// chamfer terms are reduced per block in FP64 and then in a fixed order.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "block_scan.cuh"
#include "internal.h"

namespace esim {
namespace {

constexpr int kQThreads = 256;
constexpr int kMaxTau = 16;

__global__ void esim_frame_kernel(const float* __restrict__ rad, int channels, float log_eps, float C,
                                  int init, float* __restrict__ l_last, int32_t* __restrict__ counts,
                                  long long n)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float Y = channels == 3
            ? 0.2126f * __ldg(rad + i) + 0.7152f * __ldg(rad + n + i) + 0.0722f * __ldg(rad + 2 * n + i)
            : __ldg(rad + i);
        const float y = logf(Y + log_eps);
        if (init) {
            l_last[i] = y;
            counts[i] = 0;
            continue;
        }
        const float L = l_last[i];
        const float dl = y - L;
        const float nf = floorf(fabsf(dl) / C);
        if (nf >= 1.0f) {
            const float pol = dl > 0.0f ? 1.0f : -1.0f;
            l_last[i] = fmaf(pol * nf, C, L);
            counts[i] = (int32_t)(pol * nf);
        } else {
            counts[i] = 0;
        }
    }
}

constexpr int kColumns = 32;             // image columns of a column-pass block
constexpr int kMaxRows = 4096;           // rows whose event masks that block holds
constexpr int kRowChunkBytes = 16 * kColumns;   // masks and carried rows of 32 rows, both polarities
constexpr int kQueryThreads = 128;
constexpr int kQueryPix = 32 * kQueryThreads;   // pixels of a query block

struct QualParams {
    const int32_t* set[2];   // 0: generated, 1: reference; [F][H][W]
    void* g;                 // [set][polarity][F][H][W] rows to the nearest event of the column (max: none)
    uint32_t* frame_any;     // [set][polarity][F]: the frame holds an event of that polarity
    unsigned long long* hit; // [direction][kMaxTau] event counts within tau
    unsigned long long* n_ev;   // [direction] events queried
    uint32_t* unmatched;     // [direction] some event had no partner of its polarity
    double* partial;         // [direction][query blocks] sums of n * d^2
    int W, H, F, n_tau;
    float invW, invH, invF;
    float tau2[kMaxTau];
    int q_blocks;
};

template <class G>
constexpr G kNoEvent = (G)~(G)0;

// Column distances of images up to kMaxRows high.  A block takes 32 columns of
// one frame: its warps read the counts once, 32 rows at a time, into one event
// mask per (column, 32 rows, polarity); one thread per column and polarity
// carries the last event down and the next one up over the masks; the warps
// then write every row's distance from its mask and the two carried rows.  It
// is bound by memory: 4 B read and 4 B written per pixel and set.  At 1280 x
// 720 x 120: 0.44 ms (0.26 at the copy rate), against 1.66 ms with one thread
// walking each column down and up (4-byte squared distances, written, read
// back and written again).
__global__ void __launch_bounds__(kQThreads) column_mask_kernel(QualParams p)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int n_chunks = (p.H + 31) / 32;
    uint32_t* mask = reinterpret_cast<uint32_t*>(sm);                                 // [polarity][chunk][column]
    short* before = reinterpret_cast<short*>(mask + 2 * n_chunks * kColumns);         // last event row above the chunk
    short* after = before + 2 * n_chunks * kColumns;                                  // first event row below it
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = blockIdx.x * kColumns + lane, t = blockIdx.y, s = blockIdx.z;
    const size_t N = (size_t)p.W * p.H;
    const int32_t* c = p.set[s] + (size_t)t * N + x;
    uint32_t any0 = 0u, any1 = 0u;
    for (int k = warp; k < n_chunks; k += kQThreads / 32) {
        uint32_t m0 = 0u, m1 = 0u;
        if (x < p.W) {
            const int rows = min(32, p.H - 32 * k);
            const int32_t* ck = c + (size_t)(32 * k) * p.W;
            if (rows == 32) {
#pragma unroll
                for (int r = 0; r < 32; ++r) {
                    const int32_t v = __ldg(ck + (size_t)r * p.W);
                    m0 |= (v > 0 ? 1u : 0u) << r;
                    m1 |= (v < 0 ? 1u : 0u) << r;
                }
            } else {
                for (int r = 0; r < rows; ++r) {
                    const int32_t v = __ldg(ck + (size_t)r * p.W);
                    m0 |= (v > 0 ? 1u : 0u) << r;
                    m1 |= (v < 0 ? 1u : 0u) << r;
                }
            }
        }
        mask[k * kColumns + lane] = m0;
        mask[(n_chunks + k) * kColumns + lane] = m1;
        any0 |= m0;
        any1 |= m1;
    }
    any0 = __reduce_or_sync(0xffffffffu, any0);
    any1 = __reduce_or_sync(0xffffffffu, any1);
    if (lane == 0 && any0) atomicOr(&p.frame_any[(2 * s + 0) * p.F + t], 1u);
    if (lane == 0 && any1) atomicOr(&p.frame_any[(2 * s + 1) * p.F + t], 1u);
    __syncthreads();
    if (threadIdx.x < 4 * kColumns) {
        // warps 0, 1: down, polarity 0, 1; warps 2, 3: up
        const int pol = warp & 1, at = pol * n_chunks * kColumns + lane;
        if (warp < 2) {
            int last = -1;
            for (int k = 0; k < n_chunks; ++k) {
                before[at + k * kColumns] = (short)last;
                const uint32_t m = mask[at + k * kColumns];
                if (m) last = 32 * k + 31 - __clz(m);
            }
        } else {
            int next = -1;
            for (int k = n_chunks - 1; k >= 0; --k) {
                after[at + k * kColumns] = (short)next;
                const uint32_t m = mask[at + k * kColumns];
                if (m) next = 32 * k + __ffs(m) - 1;
            }
        }
    }
    __syncthreads();
    if (x >= p.W) return;
    for (int k = warp; k < 2 * n_chunks; k += kQThreads / 32) {
        const int pol = k >= n_chunks ? 1 : 0, ch = k - pol * n_chunks;
        const uint32_t m = mask[k * kColumns + lane];
        const int lo = before[k * kColumns + lane], hi = after[k * kColumns + lane];
        const int rows = min(32, p.H - 32 * ch);
        unsigned short* g = static_cast<unsigned short*>(p.g) + ((size_t)(2 * s + pol) * p.F + t) * N +
                            (size_t)(32 * ch) * p.W + x;
#pragma unroll 4
        for (int r = 0; r < rows; ++r) {
            const int y = 32 * ch + r;
            const uint32_t up = m << (31 - r), down = m >> r;   // events at or above, at or below the row
            unsigned d = up ? (unsigned)__clz(up) : lo >= 0 ? (unsigned)(y - lo) : 0xffffu;
            d = min(d, down ? (unsigned)__ffs(down) - 1u : hi >= 0 ? (unsigned)(hi - y) : 0xffffu);
            g[(size_t)r * p.W] = (unsigned short)d;
        }
    }
}

// Column distances of taller images: one thread per (column, frame, set), both
// polarities, downward then upward.
__global__ void column_walk_kernel(QualParams p)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.y;
    const int s = blockIdx.z;
    if (x >= p.W) return;
    const size_t N = (size_t)p.W * p.H;
    const int32_t* c = p.set[s] + (size_t)t * N + x;
    uint32_t* g0 = static_cast<uint32_t*>(p.g) + ((size_t)(2 * s + 0) * p.F + t) * N + x;
    uint32_t* g1 = static_cast<uint32_t*>(p.g) + ((size_t)(2 * s + 1) * p.F + t) * N + x;
    int last0 = -1, last1 = -1;
    for (int y = 0; y < p.H; ++y) {
        const int32_t v = c[(size_t)y * p.W];
        if (v > 0) last0 = y;
        if (v < 0) last1 = y;
        g0[(size_t)y * p.W] = last0 < 0 ? kNoEvent<uint32_t> : (uint32_t)(y - last0);
        g1[(size_t)y * p.W] = last1 < 0 ? kNoEvent<uint32_t> : (uint32_t)(y - last1);
    }
    if (last0 >= 0) atomicOr(&p.frame_any[(2 * s + 0) * p.F + t], 1u);
    if (last1 >= 0) atomicOr(&p.frame_any[(2 * s + 1) * p.F + t], 1u);
    last0 = last1 = -1;
    for (int y = p.H - 1; y >= 0; --y) {
        const int32_t v = c[(size_t)y * p.W];
        if (v > 0) last0 = y;
        if (v < 0) last1 = y;
        if (last0 >= 0) g0[(size_t)y * p.W] = min(g0[(size_t)y * p.W], (uint32_t)(last0 - y));
        if (last1 >= 0) g1[(size_t)y * p.W] = min(g1[(size_t)y * p.W], (uint32_t)(last1 - y));
    }
}

// Squared distance from (x, y, t) to the nearest event of polarity pol in set
// s.  Columns go outward eight at a time, all their loads in flight at once
// (a column past the cut-off only offers a larger distance).
template <class G>
__device__ __forceinline__ float nearest2(const QualParams& p, int s, int pol, int x, int y, int t)
{
    constexpr int kStep = 8;
    const size_t N = (size_t)p.W * p.H;
    const uint32_t* any = p.frame_any + (2 * s + pol) * p.F;
    const G* gs = static_cast<const G*>(p.g) + (size_t)(2 * s + pol) * p.F * N + (size_t)y * p.W + x;
    float best = INFINITY;
    for (int k = 0; k < p.F; ++k) {
        const float dt = (float)k * p.invF;
        const float dt2 = dt * dt;
        if (dt2 >= best) break;
        for (int side = 0; side < (k ? 2 : 1); ++side) {
            const int tt = side ? t + k : t - k;
            if (tt < 0 || tt >= p.F || !any[tt]) continue;
            const G* row = gs + (size_t)tt * N;
            for (int j0 = 0; j0 < p.W; j0 += kStep) {
                const float d0 = (float)j0 * p.invW;
                if (fmaf(d0, d0, dt2) >= best) break;
                G l[kStep], r[kStep];
#pragma unroll
                for (int i = 0; i < kStep; ++i) {
                    l[i] = x - j0 - i >= 0 ? __ldg(row - j0 - i) : kNoEvent<G>;
                    r[i] = x + j0 + i < p.W ? __ldg(row + j0 + i) : kNoEvent<G>;
                }
#pragma unroll
                for (int i = 0; i < kStep; ++i) {
                    const float dx = (float)(j0 + i) * p.invW;
                    const float dy = (float)min(l[i], r[i]) * p.invH;
                    // dy^2 is rounded by itself: contracted into the sum, distances that equal
                    // a threshold would fall on its other side
                    best = fminf(best, __fadd_rn(fmaf(dx, dx, dt2), __fmul_rn(dy, dy)));
                }
            }
        }
    }
    // Two events are less than sqrt(3) apart; rows that stand for "no event" give at least 4
    // (2^32 - 1 rows of at most 2^31, 2^16 - 1 of at most 4096).
    return best < 3.5f ? best : INFINITY;
}

// 4096 pixels of the query set per block; blockIdx.y = direction (0: generated
// -> reference, 1: reference -> generated).  The block first lists its pixels
// with events, in order, so that every lane of its warps has an event to search
// for (a thread per pixel left most lanes idle: a few percent of the pixels
// have events).  A thread counts into its own slots; 64-bit shared atomics took
// most of the time of searches that end at once.  Bound by the latency of the
// searches' dependent steps.  At 1280 x 720 x 120 with 7.3 M and 6.4 M events:
// 7.35 ms with a thread per pixel, 3.27 with lists of 2048 pixels, 1.80 with
// slots in place of atomics and 1024 pixels, 1.24 with 4096 pixels and eight
// columns a step (1024 pixels: partly filled warps; 64 or 256 threads: slower).
// Small and dense sets gain too (whole evaluations, a thread per pixel -> here): 96 x
// 64 x 6 with 1% and all of the pixels 109 -> 87 and 124 -> 121 us, 160 x 120 x 10 135 -> 93 and
// 219 -> 124, 1280 x 720 x 30 2.4 -> 0.32 and 11.4 -> 1.03 ms.
template <class G>
__global__ void __launch_bounds__(kQueryThreads) query_kernel(QualParams p)
{
    constexpr int kPer = kQueryPix / kQueryThreads;
    const int dir = blockIdx.y;
    const size_t N = (size_t)p.W * p.H, total = N * (size_t)p.F;
    const size_t base = (size_t)blockIdx.x * kQueryPix;
    __shared__ unsigned short s_list[kQueryPix];
    __shared__ int s_warp[kQueryThreads / 32];
    __shared__ unsigned long long s_hit[kMaxTau][kQueryThreads];
    __shared__ unsigned long long s_n[kQueryThreads / 32];
    __shared__ double s_sum[kQueryThreads / 32];
    // one bit per pixel of the thread's run of kPer
    const size_t i0 = base + (size_t)threadIdx.x * kPer;
    const int32_t* src = p.set[dir] + i0;
    uint32_t mask = 0u;
    if (i0 + kPer <= total && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
#pragma unroll
        for (int k = 0; k < kPer / 4; ++k) {
            const int4 a = __ldg(reinterpret_cast<const int4*>(src) + k);
            mask |= ((a.x != 0 ? 1u : 0u) | (a.y != 0 ? 2u : 0u) | (a.z != 0 ? 4u : 0u) | (a.w != 0 ? 8u : 0u)) << (4 * k);
        }
    } else {
        for (int k = 0; k < kPer; ++k)
            if (i0 + k < total && __ldg(src + k) != 0) mask |= 1u << k;
    }
    int n;
    int at = block_exclusive_scan(__popc(mask), s_warp, n);
    for (; mask; mask &= mask - 1u) s_list[at++] = (unsigned short)(threadIdx.x * kPer + __ffs(mask) - 1);
    if (n == 0) {
        if (threadIdx.x == 0) p.partial[(size_t)dir * p.q_blocks + blockIdx.x] = 0.0;
        return;
    }
    for (int k = 0; k < p.n_tau; ++k) s_hit[k][threadIdx.x] = 0ull;
    __syncthreads();
    double sum = 0.0;
    unsigned long long events = 0ull;
    bool unmatched = false;
    for (int e = threadIdx.x; e < n; e += kQueryThreads) {
        const size_t idx = base + s_list[e];
        const int32_t c = __ldg(p.set[dir] + idx);
        const int t = (int)(idx / N);
        const int rem = (int)(idx - (size_t)t * N);
        const int y = rem / p.W, x = rem - y * p.W;
        const unsigned long long w = (unsigned long long)(c > 0 ? (long long)c : -(long long)c);
        const float d2 = nearest2<G>(p, 1 - dir, c > 0 ? 0 : 1, x, y, t);
        events += w;
        if (isinf(d2)) {
            unmatched = true;
        } else {
            sum += (double)w * (double)d2;
            for (int k = 0; k < p.n_tau; ++k)
                if (d2 < p.tau2[k]) s_hit[k][threadIdx.x] += w;
        }
    }
    if (unmatched) atomicOr(&p.unmatched[dir], 1u);
    // block sums in a fixed order
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        sum += __shfl_down_sync(0xffffffffu, sum, off);
        events += __shfl_down_sync(0xffffffffu, events, off);
    }
    if (lane == 0) {
        s_sum[warp] = sum;
        s_n[warp] = events;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0;
        unsigned long long m = 0ull;
        for (int i = 0; i < kQueryThreads / 32; ++i) {
            b += s_sum[i];
            m += s_n[i];
        }
        p.partial[(size_t)dir * p.q_blocks + blockIdx.x] = b;
        atomicAdd(&p.n_ev[dir], m);
    }
    for (int k = warp; k < p.n_tau; k += kQueryThreads / 32) {
        unsigned long long h = 0ull;
#pragma unroll
        for (int i = 0; i < kQueryThreads / 32; ++i) h += s_hit[k][32 * i + lane];
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) h += __shfl_down_sync(0xffffffffu, h, off);
        if (lane == 0 && h) atomicAdd(&p.hit[dir * kMaxTau + k], h);
    }
}

// Fixed-order sum of the per-block partials, one block per direction.
__global__ void __launch_bounds__(1024) reduce_kernel(QualParams p, double* out)
{
    __shared__ double s[1024];
    const double* in = p.partial + (size_t)blockIdx.x * p.q_blocks;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = threadIdx.x; i < p.q_blocks; i += 4096)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + 1024 * k < p.q_blocks) acc[k] += in[i + 1024 * k];
    s[threadIdx.x] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    __syncthreads();
    for (int w = 512; w >= 1; w >>= 1) {
        if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = s[0];
}

struct QualLayout {
    size_t g, any, hit, n_ev, unmatched, partial, sums, total;
};

QualLayout qual_layout(int W, int H, int F)
{
    const size_t N = (size_t)W * H;
    const size_t q_blocks = (N * (size_t)F + kQThreads - 1) / kQThreads;
    QualLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off = (off + bytes + 255) & ~(size_t)255;
        return at;
    };
    L.g = take(4 * (size_t)F * N * sizeof(uint32_t));   // half of it used by images up to kMaxRows high
    L.any = take(4 * (size_t)F * sizeof(uint32_t));
    L.hit = take(2 * kMaxTau * sizeof(unsigned long long));
    L.n_ev = take(2 * sizeof(unsigned long long));
    L.unmatched = take(2 * sizeof(uint32_t));
    L.partial = take(2 * q_blocks * sizeof(double));
    L.sums = take(2 * sizeof(double));
    L.total = off;
    return L;
}

}  // namespace
}  // namespace esim

using namespace esim;

extern "C" esim_ad_status esim_ad_esim_frame(const float* radiance, int32_t channels, float log_eps,
                                             float contrast, int32_t init, float* l_last, int32_t* counts,
                                             int64_t n_pix, void* cuda_stream)
{
    if (!radiance || !l_last || !counts || (channels != 1 && channels != 3) || n_pix < 0 ||
        !(contrast > 0.0f))
        return ESIM_AD_EINVAL;
    if (n_pix == 0) return ESIM_AD_OK;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return ESIM_AD_ECUDA;
    const long long blocks = (n_pix + 255) / 256;
    const int grid = (int)(blocks < (long long)sms * 16 ? blocks : (long long)sms * 16);
    esim_frame_kernel<<<grid, 256, 0, (cudaStream_t)cuda_stream>>>(radiance, channels, log_eps, contrast, init,
                                                                  l_last, counts, (long long)n_pix);
    return cudaGetLastError() == cudaSuccess ? ESIM_AD_OK : ESIM_AD_ECUDA;
}

extern "C" size_t esim_ad_quality_workspace_size(int32_t width, int32_t height, int32_t frames)
{
    if (width <= 0 || height <= 0 || frames <= 0) return 0;
    return qual_layout(width, height, frames).total;
}

extern "C" esim_ad_status esim_ad_quality(const int32_t* gen, const int32_t* ref, int32_t width, int32_t height,
                                          int32_t frames, const float* tau, int32_t n_tau, void* workspace,
                                          size_t workspace_bytes, esim_ad_quality_result* out, void* cuda_stream)
{
    if (!gen || !ref || !tau || !workspace || !out || width <= 0 || height <= 0 || frames <= 0 || frames > 65535 || n_tau < 1 ||
        n_tau > kMaxTau)
        return ESIM_AD_EINVAL;
    const QualLayout L = qual_layout(width, height, frames);
    if (workspace_bytes < L.total) return ESIM_AD_EINVAL;
    const size_t N = (size_t)width * height;
    if ((N * (size_t)frames + kQThreads - 1) / kQThreads > 0x7fffffffu) return ESIM_AD_EINVAL;
    const size_t q_blocks = (N * (size_t)frames + kQueryPix - 1) / kQueryPix;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    QualParams p;
    p.set[0] = gen;
    p.set[1] = ref;
    p.g = ws + L.g;
    p.frame_any = reinterpret_cast<uint32_t*>(ws + L.any);
    p.hit = reinterpret_cast<unsigned long long*>(ws + L.hit);
    p.n_ev = reinterpret_cast<unsigned long long*>(ws + L.n_ev);
    p.unmatched = reinterpret_cast<uint32_t*>(ws + L.unmatched);
    p.partial = reinterpret_cast<double*>(ws + L.partial);
    p.W = width;
    p.H = height;
    p.F = frames;
    p.n_tau = n_tau;
    p.invW = 1.0f / (float)width;
    p.invH = 1.0f / (float)height;
    p.invF = 1.0f / (float)frames;
    for (int k = 0; k < kMaxTau; ++k) p.tau2[k] = k < n_tau ? tau[k] * tau[k] : 0.0f;
    p.q_blocks = (int)q_blocks;
    // counters (everything between the flags and the partials) start at zero
    if (cudaMemsetAsync(ws + L.any, 0, L.partial - L.any, s) != cudaSuccess) return ESIM_AD_ECUDA;
    const bool masks = height <= kMaxRows;
    if (masks) {
        // an image up to kMaxRows high keeps its masks in shared memory, and its distances fit 16 bits
        const int smem = (height + 31) / 32 * kRowChunkBytes;
        // the limit that every call needs at most: it is the process's, and other threads set it too
        if (smem > 48 * 1024 && cudaFuncSetAttribute(column_mask_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     kMaxRows / 32 * kRowChunkBytes) != cudaSuccess)
            return ESIM_AD_ECUDA;
        column_mask_kernel<<<dim3((width + kColumns - 1) / kColumns, frames, 2), kQThreads, smem, s>>>(p);
    } else {
        column_walk_kernel<<<dim3((width + 127) / 128, frames, 2), 128, 0, s>>>(p);
    }
    if (cudaGetLastError() != cudaSuccess) return ESIM_AD_ECUDA;
    if (masks)
        query_kernel<unsigned short><<<dim3((unsigned)q_blocks, 2), kQueryThreads, 0, s>>>(p);
    else
        query_kernel<uint32_t><<<dim3((unsigned)q_blocks, 2), kQueryThreads, 0, s>>>(p);
    if (cudaGetLastError() != cudaSuccess) return ESIM_AD_ECUDA;
    double* sums = reinterpret_cast<double*>(ws + L.sums);
    reduce_kernel<<<2, 1024, 0, s>>>(p, sums);
    if (cudaGetLastError() != cudaSuccess) return ESIM_AD_ECUDA;
    unsigned long long h_hit[2 * kMaxTau], h_n[2];
    uint32_t h_un[2];
    double h_sum[2];
    if (cudaMemcpyAsync(h_hit, p.hit, sizeof(h_hit), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(h_n, p.n_ev, sizeof(h_n), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(h_un, p.unmatched, sizeof(h_un), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(h_sum, sums, sizeof(h_sum), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return ESIM_AD_ECUDA;
    esim_ad_quality_result r;
    memset(&r, 0, sizeof(r));
    r.n_tau = n_tau;
    r.n_gen = h_n[0];
    r.n_ref = h_n[1];
    for (int k = 0; k < n_tau; ++k) {
        r.tau[k] = tau[k];
        const double P = h_n[0] ? (double)h_hit[k] / (double)h_n[0] : 0.0;
        const double R = h_n[1] ? (double)h_hit[kMaxTau + k] / (double)h_n[1] : 0.0;
        r.precision[k] = P;
        r.recall[k] = R;
        r.fscore[k] = P + R > 0.0 ? 2.0 * P * R / (P + R) : 0.0;
    }
    if (h_un[0] || h_un[1]) {
        r.chamfer = INFINITY;
    } else {
        r.chamfer = (h_n[0] ? h_sum[0] / (double)h_n[0] : 0.0) + (h_n[1] ? h_sum[1] / (double)h_n[1] : 0.0);
    }
    *out = r;
    return ESIM_AD_OK;
}
