// Differentiation form: dense weighted local regression over a sequence and its
// adjoint (backward) with respect to the noisy radiance and the seven feature
// bandwidths of Eq. 5.
//
// Forward, per frame t and centre c: the regression of Eqs. 3-5 over frames
// t-T+1..t (same arithmetic as the simulator: scaled regressors
// u = s * d with s = k / (h b), w = 2^-|u|^2, FP32 Gram, equilibrated Cholesky),
// keeping theta' and v' = A'^-1 e_0 in the scaled basis.
//
// Backward (adjoint of alpha = e_0^T A^-1 g):
//   d alpha / d y_i = w_i v^T z_i
//   d alpha / d w_i = v^T z_i r_i - lambda v^T P theta     (ridge lambda W |beta|^2)
//   d w_i / d b_j   = w_i d_ij^2 / (h^2 b_j^3) = w_i u_ij^2 / (k^2 b_j)
//   d y / d E_ch    = lum_ch / (Y + eps)
// where v^T z_i = v'^T u_i in the scaled basis and v^T P theta =
// sum_{j>=1} s_j^2 v'_j theta'_j.  The bandwidth gradient is a per-centre sum
// reduced per block into partials and then in a fixed order.  The radiance
// gradient of a pixel is a sum over the centres whose windows contain it: each
// centre tile sums its own centres' shares per neighbour (bwd_center_kernel),
// and bwd_gather_kernel adds the tiles; for windows whose tile sums exceed the
// workspace, bwd_center_gv_kernel and bwd_source_kernel gather over the centres
// instead.  Every sum has a fixed order, so every result is deterministic.
#include "esim_ad.h"
#include "internal.h"
#include "wlr_math.cuh"

namespace esim {
namespace {

constexpr double kExp2ScaleD = 0.84932180028801904272;   // sqrt(log2(e) / 2)
constexpr float kExp2Scale = 0.84932180028801904272f;

struct AdjParams {
    int W, H, F, r, T, tiles_x, rgb;
    float h, log_eps, ridge;
    const float* radiance;   // [F][C][H][W]
    const float* features;   // [F][7][H][W]
    const float* bandwidth;  // [7]
    const float4* packed;    // [F][2][H][W]: (y, normal xyz), (depth, albedo rgb)
    float* alpha;            // [F][H][W]
    float* saved;            // [F][20][H][W]: theta' (10), v' (10)
    const float* g_alpha;    // [F][H][W]
    float4* gv;              // [F][3][H][W]: g_alpha * v' (10) + 2 pad, or, in its place:
    float* part;             // [F][tiles][T][8 + 2r][32 + 2r]: a tile's shares of dL/dy per frame and neighbour
    int tiles_y;
    float* partials;         // [blocks][8]
    float* g_radiance;       // [F][C][H][W]
    float* g_bandwidth;      // [7]
};

// Regressor scales from the bandwidths (device memory, read per block).
__device__ __forceinline__ void scales(const AdjParams& p, float (&sf)[7], float& s_c, float& s_px)
{
#pragma unroll
    for (int j = 0; j < 7; ++j) sf[j] = kExp2Scale / (p.h * p.bandwidth[j]);
    s_c = kExp2Scale / p.h;
    s_px = s_c / (float)p.r;
}

__global__ void __launch_bounds__(kTilePix) pack_kernel(AdjParams p)
{
    const size_t N = (size_t)p.W * p.H;
    const int f = blockIdx.y;
    const int x = (blockIdx.x % p.tiles_x) * kTileX + (threadIdx.x & 31);
    const int y = (blockIdx.x / p.tiles_x) * kTileY + (threadIdx.x >> 5);
    if (x >= p.W || y >= p.H) return;
    const size_t i = (size_t)y * p.W + x;
    const float* rad = p.radiance + (size_t)f * (p.rgb ? 3 : 1) * N;
    const float Y = p.rgb ? 0.2126f * rad[i] + 0.7152f * rad[N + i] + 0.0722f * rad[2 * N + i] : rad[i];
    const float* ft = p.features + (size_t)f * 7 * N;
    float4* out = const_cast<float4*>(p.packed) + (size_t)f * 2 * N;
    out[i] = make_float4(logf(Y + p.log_eps), ft[i], ft[N + i], ft[2 * N + i]);
    out[N + i] = make_float4(ft[3 * N + i], ft[4 * N + i], ft[5 * N + i], ft[6 * N + i]);
}

// Equilibrated Cholesky of the ridged system; theta' = A'^-1 g and v' = A'^-1 e_0.
__device__ __forceinline__ void solve_theta_v(Acc& a, const float (&s2)[NZ], float ridge,
                                              float (&theta)[NZ], float (&v)[NZ])
{
    const float Wsum = a.G[0];
#pragma unroll
    for (int j = 1; j < NZ; ++j) a.G[tri(j, j)] = fmaf(ridge * Wsum, s2[j], a.G[tri(j, j)]);
    float dsc[NZ];
#pragma unroll
    for (int i = 0; i < NZ; ++i) dsc[i] = rsqrtf(a.G[tri(i, i)]);
#pragma unroll
    for (int i = 0; i < NZ; ++i) {
#pragma unroll
        for (int j = 0; j <= i; ++j) a.G[tri(i, j)] *= dsc[i] * dsc[j];
        a.B[i] *= dsc[i];
    }
    float inv[NZ];
#pragma unroll
    for (int j = 0; j < NZ; ++j) {
        float sj = a.G[tri(j, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) sj = fmaf(-a.G[tri(j, k)], a.G[tri(j, k)], sj);
        sj = fmaxf(sj, 1e-20f);
        const float l = sqrtf(sj);
        inv[j] = 1.0f / l;
#pragma unroll
        for (int i = j + 1; i < NZ; ++i) {
            float x = a.G[tri(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) x = fmaf(-a.G[tri(i, k)], a.G[tri(j, k)], x);
            a.G[tri(i, j)] = x * inv[j];
        }
    }
    float rhs[2][NZ];
#pragma unroll
    for (int i = 0; i < NZ; ++i) {
        rhs[0][i] = a.B[i];
        rhs[1][i] = i == 0 ? dsc[0] : 0.0f;
    }
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        float z[NZ], x[NZ];
#pragma unroll
        for (int i = 0; i < NZ; ++i) {
            float t = rhs[m][i];
#pragma unroll
            for (int k = 0; k < i; ++k) t = fmaf(-a.G[tri(i, k)], z[k], t);
            z[i] = t * inv[i];
        }
#pragma unroll
        for (int i = NZ - 1; i >= 0; --i) {
            float t = z[i];
#pragma unroll
            for (int k = i + 1; k < NZ; ++k) t = fmaf(-a.G[tri(k, i)], x[k], t);
            x[i] = t * inv[i];
        }
#pragma unroll
        for (int i = 0; i < NZ; ++i) {
            if (m == 0) theta[i] = x[i] * dsc[i];
            else v[i] = x[i] * dsc[i];
        }
    }
}

// Sums of the normal equations in packed FP32 pairs (a packed FMA rounds each half
// as a single one does), regressors in pairs U_k = (u_2k, u_2k+1), u_0 = 1.  Per
// neighbour w U_k is rounded first, then multiplied into the running sums: column
// j of the Gram's triangle from row 2k on takes (w U_k) * u_j, and what is left over
// are the diagonal entries of odd rows.
struct FwdSums {
    float2 g[25];   // column 0: rows 0-9; columns 1, 2: rows 2-9; 3, 4: rows 4-9; 5, 6: rows 6-9; 7, 8: rows 8, 9
    float d[5];     // rows and columns 1, 3, 5, 7, 9
    float2 b[5];
};

// First pair of column j, and the row it starts at.
__host__ __device__ constexpr int fwd_row(int j) { return (j + 1) & ~1; }
__host__ __device__ constexpr int fwd_pair(int j)
{
    int n = 0;
    for (int c = 0; c < j; ++c) n += (NZ - fwd_row(c)) / 2;
    return n;
}

__device__ __forceinline__ void fwd_add(FwdSums& a, const float4 h0, const float4 h1, float u1, float u2, float en0,
                                        float snx, float cnx, const float2 (&sc)[3], const float2 (&nc)[3])
{
    float2 U[5];
    const float unx = fmaf(h0.y, snx, -cnx);
    U[0] = make_float2(1.0f, u1);
    U[1] = make_float2(u2, unx);
    U[2] = __ffma2_rn(make_float2(h0.z, h0.w), sc[0], nc[0]);
    U[3] = __ffma2_rn(make_float2(h1.x, h1.y), sc[1], nc[1]);
    U[4] = __ffma2_rn(make_float2(h1.z, h1.w), sc[2], nc[2]);
    float en = fmaf(-unx, unx, en0);
#pragma unroll
    for (int k = 2; k < 5; ++k) {
        en = fmaf(-U[k].x, U[k].x, en);
        en = fmaf(-U[k].y, U[k].y, en);
    }
    const float w = ex2_approx(en), wy = w * h0.x;
    float2 wU[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        wU[k] = __fmul2_rn(make_float2(w, w), U[k]);
        a.b[k] = __ffma2_rn(make_float2(wy, wy), U[k], a.b[k]);
        a.g[k] = __fadd2_rn(a.g[k], wU[k]);
        a.d[k] = fmaf(wU[k].y, U[k].y, a.d[k]);
    }
#pragma unroll
    for (int j = 1; j < 9; ++j) {
        const float u = j & 1 ? U[j / 2].y : U[j / 2].x;
#pragma unroll
        for (int i = fwd_row(j); i < NZ; i += 2) {
            const int k = fwd_pair(j) + (i - fwd_row(j)) / 2;
            a.g[k] = __ffma2_rn(wU[i / 2], make_float2(u, u), a.g[k]);
        }
    }
}

// One thread per pixel, 32 x 4 pixels per CTA.  FP32-bound: 65% of the FMA
// pipe at 16 warps per SM.  512 x 512 x 16, 7 x 7 x 3 window: 2.11 ms, against
// 2.25 ms with single FMAs and 32 x 8 pixels (2.18 packed, 2.15 with the
// record loaded ahead).  Summing over the frames at each offset before the
// coordinates are multiplied in takes fewer operations (2.11 ms unpacked) but
// left the bandwidth gradient 1.6 times as far from float64.
constexpr int kFwdThreads = 128, kFwdTileY = kFwdThreads / kTileX;

__global__ void __launch_bounds__(kFwdThreads, 4) fwd_kernel(AdjParams p)
{
    const size_t N = (size_t)p.W * p.H;
    const int f = blockIdx.y;
    const int cx = (blockIdx.x % p.tiles_x) * kTileX + (threadIdx.x & 31);
    const int cy = (blockIdx.x / p.tiles_x) * kFwdTileY + (threadIdx.x >> 5);
    if (cx >= p.W || cy >= p.H) return;
    float sf[7], s_c, s_px;
    scales(p, sf, s_c, s_px);
    const size_t ci = (size_t)cy * p.W + cx;
    const float4 c0 = p.packed[(size_t)f * 2 * N + ci];
    const float4 c1 = p.packed[((size_t)f * 2 + 1) * N + ci];
    const float cnx = c0.y * sf[0];
    const float2 sc[3] = {make_float2(sf[1], sf[2]), make_float2(sf[3], sf[4]), make_float2(sf[5], sf[6])};
    const float2 nc[3] = {make_float2(-(c0.z * sf[1]), -(c0.w * sf[2])), make_float2(-(c1.x * sf[3]), -(c1.y * sf[4])),
                          make_float2(-(c1.z * sf[5]), -(c1.w * sf[6]))};
    FwdSums sum;
#pragma unroll
    for (int i = 0; i < 25; ++i) sum.g[i] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        sum.b[i] = make_float2(0.0f, 0.0f);
        sum.d[i] = 0.0f;
    }
    const int dxlo = max(-p.r, -cx), dxhi = min(p.r, p.W - 1 - cx);
    const int dylo = max(-p.r, -cy), dyhi = min(p.r, p.H - 1 - cy);
    const int tau0 = max(0, f - p.T + 1);
    for (int tau = tau0; tau <= f; ++tau) {
        const float4* P = p.packed + (size_t)tau * 2 * N + ci;
        for (int oy = dylo; oy <= dyhi; ++oy) {
            const float u2 = (float)oy * s_px;
            // the next neighbour's record is loaded a step ahead (the row's last, once more)
            const float4* q = P + (oy * p.W + dxlo);
            float4 n0 = __ldg(q), n1 = __ldg(q + N);
#pragma unroll 1
            for (int ox = dxlo; ox <= dxhi; ++ox) {
                const float u1 = (float)ox * s_px;
                const float4 h0 = n0, h1 = n1;
                q += ox < dxhi ? 1 : 0;
                n0 = __ldg(q);
                n1 = __ldg(q + N);
                fwd_add(sum, h0, h1, u1, u2, -fmaf(u1, u1, u2 * u2), sf[0], cnx, sc, nc);
            }
        }
    }
    Acc acc;
#pragma unroll
    for (int j = 0; j < 9; ++j)
#pragma unroll
        for (int i = fwd_row(j); i < NZ; ++i) {
            const float2 v = sum.g[fwd_pair(j) + (i - fwd_row(j)) / 2];
            acc.G[tri(i, j)] = i & 1 ? v.y : v.x;
        }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        acc.G[tri(2 * k + 1, 2 * k + 1)] = sum.d[k];
        acc.B[2 * k] = sum.b[k].x;
        acc.B[2 * k + 1] = sum.b[k].y;
    }
    float s2[NZ];
    s2[0] = 0.0f;
    s2[1] = s_c * s_c;
    s2[2] = s2[1];
#pragma unroll
    for (int j = 0; j < 7; ++j) s2[3 + j] = sf[j] * sf[j];
    float theta[NZ], v[NZ];
    solve_theta_v(acc, s2, p.ridge, theta, v);
    p.alpha[(size_t)f * N + ci] = theta[0];
    float* sv = p.saved + (size_t)f * 20 * N + ci;
#pragma unroll
    for (int k = 0; k < NZ; ++k) {
        sv[(size_t)k * N] = theta[k];
        sv[(size_t)(NZ + k) * N] = v[k];
    }
}

constexpr int kCtrRows = 2;
constexpr int kCtrThreads = kTilePix / kCtrRows;
constexpr int kCtrWarps = kCtrThreads / 32;

// A block's share of the bandwidth gradient: tree sum in a fixed order -> one partial per block.
__device__ __forceinline__ void store_partial(const AdjParams& p, const float (&gb)[7])
{
    __shared__ float red[kCtrThreads][8];
#pragma unroll
    for (int j = 0; j < 7; ++j) red[threadIdx.x][j] = gb[j];
    __syncthreads();
    for (int s = kCtrThreads / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s)
#pragma unroll
            for (int j = 0; j < 7; ++j) red[threadIdx.x][j] += red[threadIdx.x + s][j];
        __syncthreads();
    }
    if (threadIdx.x < 7)
        p.partials[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 8 + threadIdx.x] = red[0][threadIdx.x];
}

// Per centre: its share of the bandwidth gradient (sum over its window of
// g_alpha (d alpha/d w_i) w_i u_ij^2), and g_alpha v'^T u_i w_i, its share of its
// neighbours' dL/dy.  Each thread takes two centres stacked in one column, so
// every neighbour record it loads (32 bytes) serves both, and the two run as
// one stream of packed FP32 pairs: 63 instructions per record instead of 70 per
// pair.  Rows that lie in one centre's window only are left out of the other's
// sums, and so are centres that the loss leaves out.
// A 128-thread CTA covers one 32 x 8 tile.
//
// At each offset the lanes' shares go to neighbouring columns of one row;
// a rotation by the offset brings them to the lane of their column (what
// wraps around belongs to the halo on the other side).  A warp's rows are
// summed in registers over the offsets, the tile's warps in shared memory in
// warp order, one frame of the window at a time.
//
// 512 x 512 x 16, 7 x 7 x 3 window: 1.80 ms and 0.13 ms for the gather, against
// 1.51 ms and 1.08 ms for bwd_source_kernel (1.93 without loading a record ahead);
// the FMA pipe is 53% busy, and most stalls are waits on the previous result.
__global__ void __launch_bounds__(kCtrThreads, 4) bwd_center_kernel(AdjParams p)
{
    extern __shared__ float s_rows[];   // [frame parity][warp][2r + 2][32 + 2r]
    const size_t N = (size_t)p.W * p.H;
    const int f = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ty0 = (blockIdx.x / p.tiles_x) * kTileY;
    const int cx = (blockIdx.x % p.tiles_x) * kTileX + lane;
    const int cy0 = ty0 + kCtrRows * warp;
    float sf[7], s_c, s_px;
    scales(p, sf, s_c, s_px);
    // the two centres' quantities side by side; zeros (and g_alpha = 0) outside the image
    float ga[2], lvpt[2], t0[2][NZ], v0[2][NZ], c0[2][7];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int cy = cy0 + k;
        ga[k] = 0.0f;
        lvpt[k] = 0.0f;
#pragma unroll
        for (int i = 0; i < NZ; ++i) t0[k][i] = v0[k][i] = 0.0f;
#pragma unroll
        for (int j = 0; j < 7; ++j) c0[k][j] = 0.0f;
        if (cx >= p.W || cy >= p.H) continue;
        const size_t ci = (size_t)cy * p.W + cx;
        ga[k] = p.g_alpha[(size_t)f * N + ci];
        if (ga[k] != 0.0f) {   // a centre that the loss leaves out adds nothing, whatever was solved there
            const float* sv = p.saved + (size_t)f * 20 * N + ci;
#pragma unroll
            for (int i = 0; i < NZ; ++i) {
                t0[k][i] = sv[(size_t)i * N];
                v0[k][i] = sv[(size_t)(NZ + i) * N];
            }
        }
        // lambda v^T P theta in natural units
        float vpt = (s_c * s_c) * (v0[k][1] * t0[k][1] + v0[k][2] * t0[k][2]);
#pragma unroll
        for (int j = 0; j < 7; ++j) vpt = fmaf(sf[j] * sf[j], v0[k][3 + j] * t0[k][3 + j], vpt);
        lvpt[k] = p.ridge * vpt;
        const float4 a = p.packed[(size_t)f * 2 * N + ci], b = p.packed[((size_t)f * 2 + 1) * N + ci];
        const float xc[7] = {a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int j = 0; j < 7; ++j) c0[k][j] = -(xc[j] * sf[j]);
    }
    const bool any = __any_sync(0xffffffffu, ga[0] != 0.0f || ga[1] != 0.0f);
    const float2 g2 = make_float2(ga[0], ga[1]), l2 = make_float2(-lvpt[0], -lvpt[1]);
    float2 th[NZ], v[NZ], gb[7];
#pragma unroll
    for (int i = 0; i < NZ; ++i) {
        th[i] = make_float2(-t0[0][i], -t0[1][i]);   // negated: y - fit is one sum
        v[i] = make_float2(v0[0][i], v0[1][i]);
    }
#pragma unroll
    for (int j = 0; j < 7; ++j) gb[j] = make_float2(0.0f, 0.0f);
    const int span = kTileX + 2 * p.r, rows = kCtrRows + 2 * p.r;
    float* buf = s_rows;
    for (int tau = max(0, f - p.T + 1); tau <= f; ++tau) {
        const float4* P0 = p.packed + (size_t)tau * 2 * N;
        for (int k = 0; k < rows; ++k) {
            const int ny = cy0 - p.r + k;
            if (ny < 0 || ny >= p.H) continue;
            float main_sum = 0.0f, halo_sum = 0.0f;
            if (any) {
                const float2 u2 = make_float2((float)(k - p.r) * s_px, (float)(k - p.r - 1) * s_px);
                const float2 e2 = make_float2(-(u2.x * u2.x), -(u2.y * u2.y));
                // the centres that take part: in the loss, and the row in their window
                const bool in0 = ga[0] != 0.0f && k <= 2 * p.r, in1 = ga[1] != 0.0f && k >= 1;
                const bool plain = __all_sync(0xffffffffu, in0 && in1);
                const float2 fit_row = __ffma2_rn(th[2], u2, th[0]), vz_row = __ffma2_rn(v[2], u2, v[0]);
                const float4* row = P0 + (size_t)ny * p.W + cx;
                // the next neighbour's record is loaded a step ahead
                float4 n0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), n1 = n0;
                if ((unsigned)(cx - p.r) < (unsigned)p.W) {
                    n0 = __ldg(row - p.r);
                    n1 = __ldg(row + N - p.r);
                }
#pragma unroll 1
                for (int ox = -p.r; ox <= p.r; ++ox) {
                    float share = 0.0f;
                    const float4 h0 = n0, h1 = n1;
                    if (ox < p.r && (unsigned)(cx + ox + 1) < (unsigned)p.W) {
                        n0 = __ldg(row + ox + 1);
                        n1 = __ldg(row + N + ox + 1);
                    }
                    if ((unsigned)(cx + ox) < (unsigned)p.W) {
                        const float fv[7] = {h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
                        const float u1 = (float)ox * s_px;
                        const float2 uu = make_float2(u1, u1);
                        float2 u[7], sq = make_float2(0.0f, 0.0f);
                        float2 res = __ffma2_rn(th[1], uu, fit_row), vz = __ffma2_rn(v[1], uu, vz_row);
#pragma unroll
                        for (int j = 0; j < 7; ++j) {
                            u[j] = make_float2(fmaf(fv[j], sf[j], c0[0][j]), fmaf(fv[j], sf[j], c0[1][j]));
                            sq = j ? __ffma2_rn(u[j], u[j], sq) : __fmul2_rn(u[j], u[j]);
                            res = __ffma2_rn(th[3 + j], u[j], res);
                            vz = __ffma2_rn(v[3 + j], u[j], vz);
                        }
                        const float en1 = u1 * u1;
                        const float2 w = make_float2(ex2_approx((e2.x - en1) - sq.x), ex2_approx((e2.y - en1) - sq.y));
                        const float2 gw = __fmul2_rn(g2, w);
                        res = __fadd2_rn(res, make_float2(h0.x, h0.x));
                        float2 c = __fmul2_rn(gw, __ffma2_rn(vz, res, l2)), sh = __fmul2_rn(gw, vz);
                        if (!plain) {   // a weight of 0 does not cancel what is not a number
                            c = make_float2(in0 ? c.x : 0.0f, in1 ? c.y : 0.0f);
                            sh = make_float2(in0 ? sh.x : 0.0f, in1 ? sh.y : 0.0f);
                        }
#pragma unroll
                        for (int j = 0; j < 7; ++j) gb[j] = __ffma2_rn(__fmul2_rn(c, u[j]), u[j], gb[j]);
                        share = sh.x + sh.y;
                    }
                    const float got = __shfl_sync(0xffffffffu, share, (lane - ox) & 31);
                    const bool inside = (unsigned)(lane - ox) < 32u;
                    main_sum += inside ? got : 0.0f;
                    halo_sum += inside ? 0.0f : got;
                }
            }
            float* out = buf + (warp * rows + k) * span;
            out[p.r + lane] = main_sum;
            if (lane < p.r) out[p.r + kTileX + lane] = halo_sum;             // from offsets > 0
            if (lane >= kTileX - p.r) out[lane - (kTileX - p.r)] = halo_sum;   // from offsets < 0 (r <= 15)
        }
        __syncthreads();
        const int trows = kTileY + 2 * p.r;
        float* out = p.part + (((size_t)f * gridDim.x + blockIdx.x) * p.T + (f - tau)) * trows * span;
        for (int i = threadIdx.x; i < trows * span; i += kCtrThreads) {
            const int R = i / span, col = i - R * span;
            if (ty0 - p.r + R < 0 || ty0 - p.r + R >= p.H) continue;   // no such source row
            float sum = 0.0f;
#pragma unroll
            for (int w = 0; w < kCtrWarps; ++w) {
                const int k = R - kCtrRows * w;
                if (k >= 0 && k < rows) sum += buf[(w * rows + k) * span + col];
            }
            out[i] = sum;
        }
        // the next frame's rows go to the other half: no warp is two barriers behind
        buf = buf == s_rows ? s_rows + kCtrWarps * rows * span : s_rows;
    }
    const float share[7] = {gb[0].x + gb[0].y, gb[1].x + gb[1].y, gb[2].x + gb[2].y, gb[3].x + gb[3].y,
                            gb[4].x + gb[4].y, gb[5].x + gb[5].y, gb[6].x + gb[6].y};
    store_partial(p, share);
}

// The same for windows whose tile sums exceed the workspace: g_alpha v' is left for
// bwd_source_kernel, which forms every pair's weight again.  The centres one by one
// in single FMAs, out-of-image neighbours not visited.  In packed pairs, as above,
// without shares to pass on: 512 x 512 x 4, 19 x 19 x 3 window 2.20 ms for 1.97; 24 x 20 x 2,
// 31 x 31 x 1 window 116 us for 83.
__global__ void __launch_bounds__(kCtrThreads, 4) bwd_center_gv_kernel(AdjParams p)
{
    const size_t N = (size_t)p.W * p.H;
    const int f = blockIdx.y;
    const int cx = (blockIdx.x % p.tiles_x) * kTileX + (threadIdx.x & 31);
    const int cy0 = (blockIdx.x / p.tiles_x) * kTileY + kCtrRows * (threadIdx.x >> 5);
    float sf[7], s_c, s_px;
    scales(p, sf, s_c, s_px);
    float gb[7] = {0, 0, 0, 0, 0, 0, 0};
    float ga[kCtrRows], lvpt[kCtrRows], th[kCtrRows][NZ], v[kCtrRows][NZ], cf[kCtrRows][7];
    bool active[kCtrRows];
    bool any = false;
#pragma unroll
    for (int k = 0; k < kCtrRows; ++k) {
        const int cy = cy0 + k;
        active[k] = false;
        ga[k] = 0.0f;
        lvpt[k] = 0.0f;
#pragma unroll
        for (int i = 0; i < NZ; ++i) th[k][i] = v[k][i] = 0.0f;
#pragma unroll
        for (int j = 0; j < 7; ++j) cf[k][j] = 0.0f;
        if (cx >= p.W || cy >= p.H) continue;
        const size_t ci = (size_t)cy * p.W + cx;
        ga[k] = p.g_alpha[(size_t)f * N + ci];
        const float* sv = p.saved + (size_t)f * 20 * N + ci;
#pragma unroll
        for (int i = 0; i < NZ; ++i) {
            th[k][i] = sv[(size_t)i * N];
            v[k][i] = sv[(size_t)(NZ + i) * N];
        }
        // a centre that the loss leaves out adds nothing, whatever was solved there
        auto times_ga = [&](float x) { return ga[k] != 0.0f ? ga[k] * x : 0.0f; };
        float4* g = p.gv + (size_t)f * 3 * N + ci;
        g[0] = make_float4(times_ga(v[k][0]), times_ga(v[k][1]), times_ga(v[k][2]), times_ga(v[k][3]));
        g[N] = make_float4(times_ga(v[k][4]), times_ga(v[k][5]), times_ga(v[k][6]), times_ga(v[k][7]));
        g[2 * N] = make_float4(times_ga(v[k][8]), times_ga(v[k][9]), 0.0f, 0.0f);
        if (ga[k] == 0.0f) continue;
        // lambda v^T P theta in natural units
        float vpt = (s_c * s_c) * (v[k][1] * th[k][1] + v[k][2] * th[k][2]);
#pragma unroll
        for (int j = 0; j < 7; ++j) vpt = fmaf(sf[j] * sf[j], v[k][3 + j] * th[k][3 + j], vpt);
        lvpt[k] = p.ridge * vpt;
        const float4 c0 = p.packed[(size_t)f * 2 * N + ci];
        const float4 c1 = p.packed[((size_t)f * 2 + 1) * N + ci];
        cf[k][0] = c0.y * sf[0];
        cf[k][1] = c0.z * sf[1];
        cf[k][2] = c0.w * sf[2];
        cf[k][3] = c1.x * sf[3];
        cf[k][4] = c1.y * sf[4];
        cf[k][5] = c1.z * sf[5];
        cf[k][6] = c1.w * sf[6];
        active[k] = true;
        any = true;
    }
    if (any) {
        // neighbours (cx + ox, ny) inside the image, in the window of some centre row
        const int dxlo = max(-p.r, -cx), dxhi = min(p.r, p.W - 1 - cx);
        const int nylo = max(0, cy0 - p.r), nyhi = min(p.H - 1, cy0 + kCtrRows - 1 + p.r);
        for (int tau = max(0, f - p.T + 1); tau <= f; ++tau) {
            const float4* P0 = p.packed + (size_t)tau * 2 * N;
            const float4* P1 = P0 + N;
            for (int ny = nylo; ny <= nyhi; ++ny) {
                for (int ox = dxlo; ox <= dxhi; ++ox) {
                    const float u1 = (float)ox * s_px;
                    const size_t ni = (size_t)ny * p.W + cx + ox;
                    const float4 h0 = __ldg(P0 + ni), h1 = __ldg(P1 + ni);
                    const float fv[7] = {h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
#pragma unroll
                    for (int k = 0; k < kCtrRows; ++k) {
                        const int oy = ny - (cy0 + k);
                        if (!active[k] || oy < -p.r || oy > p.r) continue;
                        const float u2 = (float)oy * s_px;
                        float u[7];
                        float en = -fmaf(u1, u1, u2 * u2);
#pragma unroll
                        for (int j = 0; j < 7; ++j) {
                            u[j] = fmaf(fv[j], sf[j], -cf[k][j]);
                            en = fmaf(-u[j], u[j], en);
                        }
                        const float w = ex2_approx(en);
                        float fit = th[k][0] + th[k][1] * u1 + th[k][2] * u2;
                        float vz = v[k][0] + v[k][1] * u1 + v[k][2] * u2;
#pragma unroll
                        for (int j = 0; j < 7; ++j) {
                            fit = fmaf(th[k][3 + j], u[j], fit);
                            vz = fmaf(v[k][3 + j], u[j], vz);
                        }
                        const float dadw = fmaf(vz, h0.x - fit, -lvpt[k]);
                        const float c = ga[k] * dadw * w;
#pragma unroll
                        for (int j = 0; j < 7; ++j) gb[j] = fmaf(c, u[j] * u[j], gb[j]);
                    }
                }
            }
        }
    }
    store_partial(p, gb);
}

// dL/dE of a pixel from its dL/dy.
__device__ __forceinline__ void store_radiance_grad(const AdjParams& p, int frame, size_t i, float gy)
{
    const size_t N = (size_t)p.W * p.H;
    const float* rad = p.radiance + (size_t)frame * (p.rgb ? 3 : 1) * N;
    float* grad = p.g_radiance + (size_t)frame * (p.rgb ? 3 : 1) * N;
    if (p.rgb) {
        const float Y = 0.2126f * rad[i] + 0.7152f * rad[N + i] + 0.0722f * rad[2 * N + i];
        const float gY = gy / (Y + p.log_eps);
        grad[i] = 0.2126f * gY;
        grad[N + i] = 0.7152f * gY;
        grad[2 * N + i] = 0.0722f * gY;
    } else {
        grad[i] = gy / (rad[i] + p.log_eps);
    }
}

// Per source pixel of frame tau: the shares that the centre tiles of frames tau
// .. tau + T - 1 whose windows reach it hold for it, in tile order.
__global__ void __launch_bounds__(kTilePix) bwd_gather_kernel(AdjParams p)
{
    const int tau = blockIdx.y;
    const int x = (blockIdx.x % p.tiles_x) * kTileX + (threadIdx.x & 31);
    const int y = (blockIdx.x / p.tiles_x) * kTileY + (threadIdx.x >> 5);
    if (x >= p.W || y >= p.H) return;
    const int span = kTileX + 2 * p.r, trows = kTileY + 2 * p.r;
    const int tx0 = max(0, x - p.r) / kTileX, tx1 = min(p.W - 1, x + p.r) / kTileX;
    const int ty0 = max(0, y - p.r) / kTileY, ty1 = min(p.H - 1, y + p.r) / kTileY;
    float gy = 0.0f;
    for (int k = 0; k < p.T && tau + k < p.F; ++k)
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx) {
                const size_t tile = (size_t)(tau + k) * (p.tiles_x * p.tiles_y) + (size_t)ty * p.tiles_x + tx;
                gy += p.part[((tile * p.T + k) * trows + (y - ty * kTileY + p.r)) * span + (x - tx * kTileX + p.r)];
            }
    store_radiance_grad(p, tau, (size_t)y * p.W + x, gy);
}

// Fixed-order reduction of the per-block partials; dL/db_j = sum / (k^2 b_j).
// One block per component, in FP64: the components' sums run side by side, and
// a partial that is infinite, or a sum past FP32's range, stays what it is.
// 512 x 512 x 16 (16384 partials): 0.014 ms, against 0.13 ms with the components
// one after the other in one block.
__global__ void __launch_bounds__(kTilePix) bwd_bandwidth_kernel(AdjParams p, int n_blocks)
{
    __shared__ double red[kTilePix];
    const int j = blockIdx.x;
    double acc = 0.0;
#pragma unroll 8
    for (int b = threadIdx.x; b < n_blocks; b += kTilePix) acc += (double)p.partials[(size_t)b * 8 + j];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = kTilePix / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        p.g_bandwidth[j] = (float)(red[0] / (kExp2ScaleD * kExp2ScaleD * (double)p.bandwidth[j]));
}

// Per source pixel q of frame tau: dL/dy = sum over centres c (|c - q| <= r) of
// frames t in [tau, tau + T - 1] of g_alpha_t(c) w v'_t(c)^T u, then dL/dE.
// Each thread gathers for kSrcRows sources stacked in one column, so every
// centre record it loads (two feature records and three g_alpha v' records,
// 80 bytes) serves each of those sources whose window holds it: 2.8 pairs per
// load at r = 3 instead of one.  A CTA covers 32 columns x 32 rows.
constexpr int kSrcRows = 4;
constexpr int kSrcTileY = kSrcRows * (kTilePix / 32);

__global__ void __launch_bounds__(kTilePix, 2) bwd_source_kernel(AdjParams p)
{
    const size_t N = (size_t)p.W * p.H;
    const int tau = blockIdx.y;
    const int qx = (blockIdx.x % p.tiles_x) * kTileX + (threadIdx.x & 31);
    const int qy0 = (blockIdx.x / p.tiles_x) * kSrcTileY + kSrcRows * (threadIdx.x >> 5);
    if (qx >= p.W || qy0 >= p.H) return;
    const int nrow = min(kSrcRows, p.H - qy0);
    float sf[7], s_c, s_px;
    scales(p, sf, s_c, s_px);
    float qf[kSrcRows][7], gy[kSrcRows];
#pragma unroll
    for (int s = 0; s < kSrcRows; ++s) {
        gy[s] = 0.0f;
        const size_t qi = (size_t)(qy0 + min(s, nrow - 1)) * p.W + qx;
        const float4 q0 = p.packed[(size_t)tau * 2 * N + qi];
        const float4 q1 = p.packed[((size_t)tau * 2 + 1) * N + qi];
        qf[s][0] = q0.y * sf[0];
        qf[s][1] = q0.z * sf[1];
        qf[s][2] = q0.w * sf[2];
        qf[s][3] = q1.x * sf[3];
        qf[s][4] = q1.y * sf[4];
        qf[s][5] = q1.z * sf[5];
        qf[s][6] = q1.w * sf[6];
    }
    // centres c = q - o (o the neighbour offset of q seen from c) inside the
    // image: columns qx - ox, rows cy with |qy - cy| <= r for some source row
    const int oxlo = max(-p.r, qx - (p.W - 1)), oxhi = min(p.r, qx);
    const int cylo = max(0, qy0 - p.r), cyhi = min(p.H - 1, qy0 + nrow - 1 + p.r);
    const int t1 = min(p.F - 1, tau + p.T - 1);
    for (int t = tau; t <= t1; ++t) {
        const float4* C0 = p.packed + (size_t)t * 2 * N;
        const float4* C1 = C0 + N;
        const float4* G = p.gv + (size_t)t * 3 * N;
        for (int cy = cylo; cy <= cyhi; ++cy) {
            for (int ox = oxlo; ox <= oxhi; ++ox) {
                const float u1 = (float)ox * s_px;
                const size_t ci = (size_t)cy * p.W + (qx - ox);
                const float4 c0 = __ldg(C0 + ci), c1 = __ldg(C1 + ci);
                const float4 g0 = __ldg(G + ci), g1 = __ldg(G + N + ci), g2 = __ldg(G + 2 * N + ci);
                const float cfv[7] = {c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                for (int s = 0; s < kSrcRows; ++s) {
                    const int oy = qy0 + s - cy;   // the same for the whole warp
                    if (s >= nrow || oy < -p.r || oy > p.r) continue;
                    const float u2 = (float)oy * s_px;
                    float u[7];
                    float en = -fmaf(u1, u1, u2 * u2);
#pragma unroll
                    for (int j = 0; j < 7; ++j) {
                        u[j] = fmaf(-cfv[j], sf[j], qf[s][j]);
                        en = fmaf(-u[j], u[j], en);
                    }
                    const float w = ex2_approx(en);
                    float vz = g0.x + g0.y * u1 + g0.z * u2;
                    vz = fmaf(g0.w, u[0], vz);
                    vz = fmaf(g1.x, u[1], vz);
                    vz = fmaf(g1.y, u[2], vz);
                    vz = fmaf(g1.z, u[3], vz);
                    vz = fmaf(g1.w, u[4], vz);
                    vz = fmaf(g2.x, u[5], vz);
                    vz = fmaf(g2.y, u[6], vz);
                    gy[s] = fmaf(w, vz, gy[s]);
                }
            }
        }
    }
#pragma unroll
    for (int s = 0; s < kSrcRows; ++s) {
        if (s >= nrow) break;
        store_radiance_grad(p, tau, (size_t)(qy0 + s) * p.W + qx, gy[s]);
    }
}

bool desc_ok(const esim_ad_wlr_desc* d)
{
    return d && d->struct_size == sizeof(esim_ad_wlr_desc) && d->width >= 1 && d->height >= 1 &&
           d->sequence >= 1 && d->radius >= 1 && d->radius <= kMaxRadius && d->frames >= 1 &&
           d->frames <= kMaxFrames && (d->radiance_fmt == ESIM_AD_LUMA_F32 || d->radiance_fmt == ESIM_AD_RGB_F32) &&
           d->h > 0.0f && d->ridge > 0.0f && d->log_eps >= 0.0f;
}

struct Layout {
    size_t packed, gv, partials, total;
    int tiles_x, tiles_y, n_tiles, n_blocks;
    bool fused;   // the centre tiles' shares fit the place of g_alpha v'
};

Layout layout(const esim_ad_wlr_desc* d)
{
    Layout L;
    const size_t N = (size_t)d->width * d->height, F = (size_t)d->sequence;
    L.tiles_x = (d->width + kTileX - 1) / kTileX;
    L.tiles_y = (d->height + kTileY - 1) / kTileY;
    L.n_tiles = L.tiles_x * L.tiles_y;
    L.n_blocks = L.n_tiles * d->sequence;
    L.packed = 0;
    L.gv = L.packed + F * 2 * N * sizeof(float4);
    L.partials = L.gv + F * 3 * N * sizeof(float4);
    L.total = L.partials + (size_t)L.n_blocks * 8 * sizeof(float);
    // per centre 4 T (8 + 2r)(32 + 2r) / 256 bytes: 25 at r = 3, T = 3, of the 48 of g_alpha v'.
    // Where it fits it is the faster way: backward calls of 24 x 20 x 2 to 512 x 512 x 4, radius 1
    // to 7 with 1 to 5 frames and 15 with 1, take 0.38 to 0.77 of the time of the other way.
    L.fused = F * L.n_tiles * d->frames * (kTileY + 2 * d->radius) * (kTileX + 2 * d->radius) * sizeof(float) <=
              F * 3 * N * sizeof(float4);
    return L;
}

AdjParams params(const esim_ad_wlr_desc* d, const Layout& L, void* ws)
{
    AdjParams p;
    p.W = d->width;
    p.H = d->height;
    p.F = d->sequence;
    p.r = d->radius;
    p.T = d->frames;
    p.tiles_x = L.tiles_x;
    p.tiles_y = L.tiles_y;
    p.rgb = d->radiance_fmt == ESIM_AD_RGB_F32 ? 1 : 0;
    p.h = d->h;
    p.log_eps = d->log_eps;
    p.ridge = d->ridge;
    unsigned char* base = static_cast<unsigned char*>(ws);
    p.packed = reinterpret_cast<const float4*>(base + L.packed);
    p.gv = reinterpret_cast<float4*>(base + L.gv);
    p.part = reinterpret_cast<float*>(base + L.gv);
    p.partials = reinterpret_cast<float*>(base + L.partials);
    p.radiance = p.features = p.bandwidth = p.g_alpha = nullptr;
    p.alpha = p.saved = p.g_radiance = p.g_bandwidth = nullptr;
    return p;
}

}  // namespace
}  // namespace esim

using namespace esim;

extern "C" size_t esim_ad_wlr_workspace_size(const esim_ad_wlr_desc* d)
{
    if (!desc_ok(d)) return 0;
    return layout(d).total;
}

extern "C" esim_ad_status esim_ad_wlr_forward(const esim_ad_wlr_desc* d, const float* radiance,
                                              const float* features, const float* bandwidth, float* alpha,
                                              float* saved, void* workspace, void* cuda_stream)
{
    if (!desc_ok(d) || !radiance || !features || !bandwidth || !alpha || !saved || !workspace)
        return ESIM_AD_EINVAL;
    const Layout L = layout(d);
    AdjParams p = params(d, L, workspace);
    p.radiance = radiance;
    p.features = features;
    p.bandwidth = bandwidth;
    p.alpha = alpha;
    p.saved = saved;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const dim3 grid(L.n_tiles, d->sequence);
    pack_kernel<<<grid, kTilePix, 0, s>>>(p);
    const dim3 grid_fwd(L.tiles_x * ((d->height + kFwdTileY - 1) / kFwdTileY), d->sequence);
    fwd_kernel<<<grid_fwd, kFwdThreads, 0, s>>>(p);
    return cudaGetLastError() == cudaSuccess ? ESIM_AD_OK : ESIM_AD_ECUDA;
}

extern "C" esim_ad_status esim_ad_wlr_backward(const esim_ad_wlr_desc* d, const float* radiance,
                                               const float* features, const float* bandwidth,
                                               const float* saved, const float* g_alpha, float* g_radiance,
                                               float* g_bandwidth, void* workspace, void* cuda_stream)
{
    if (!desc_ok(d) || !radiance || !features || !bandwidth || !saved || !g_alpha || !g_radiance ||
        !g_bandwidth || !workspace)
        return ESIM_AD_EINVAL;
    const Layout L = layout(d);
    AdjParams p = params(d, L, workspace);
    p.radiance = radiance;
    p.features = features;
    p.bandwidth = bandwidth;
    p.saved = const_cast<float*>(saved);
    p.g_alpha = g_alpha;
    p.g_radiance = g_radiance;
    p.g_bandwidth = g_bandwidth;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const dim3 grid(L.n_tiles, d->sequence);
    if (L.fused) {
        const int smem = 2 * kCtrWarps * (kCtrRows + 2 * d->radius) * (kTileX + 2 * d->radius) * (int)sizeof(float);
        if (smem > 40 * 1024 && cudaFuncSetAttribute(bwd_center_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     64 * 1024) != cudaSuccess)
            return ESIM_AD_ECUDA;
        bwd_center_kernel<<<grid, kCtrThreads, smem, s>>>(p);
    } else {
        bwd_center_gv_kernel<<<grid, kCtrThreads, 0, s>>>(p);
    }
    bwd_bandwidth_kernel<<<7, kTilePix, 0, s>>>(p, L.n_blocks);
    if (L.fused) {
        bwd_gather_kernel<<<grid, kTilePix, 0, s>>>(p);
    } else {
        const dim3 grid_src(L.tiles_x * ((d->height + kSrcTileY - 1) / kSrcTileY), d->sequence);
        bwd_source_kernel<<<grid_src, kTilePix, 0, s>>>(p);
    }
    return cudaGetLastError() == cudaSuccess ? ESIM_AD_OK : ESIM_AD_ECUDA;
}
