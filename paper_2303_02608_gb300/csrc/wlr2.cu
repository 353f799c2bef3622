// Second-order form: the dense weighted local regression of Eqs. 4-5 with the
// Taylor expansion of Eq. 3 carried one order further (the non-linear
// regression that Section 4 names as the extension).  Per frame t and centre c
// the design row of neighbour i is built from the scaled offset u = s d
// (s_j = k / (h b_j), k = sqrt(log2(e) / 2), so w = 2^-|u|^2 is the product
// Gaussian of Eq. 5):
//
//     z = (u_a u_b for a <= b [45], u [9], 1),   55 unknowns,
//
// and the log brightness y rides along as a 56th entry, so one symmetric
// 56 x 56 Gram G = sum_i w_i [z;y][z;y]^T holds the normal matrix and the
// right-hand side.  The ridge lambda W |theta_k|^2 on every coefficient but the
// intercept is added in natural units (lambda W s_a^2 s_b^2 on the diagonal of
// a quadratic unknown, lambda W s_a^2 on a linear one).  With the intercept
// ordered last among the unknowns, the upper Cholesky factor U of the augmented
// (equilibrated) Gram gives alpha = U[54][55] / U[54][54] directly: no back
// substitution.
//
// Moments.  Entry (u_a u_b, u_c u_d) of the Gram is the weighted moment of the
// monomial u_a u_b u_c u_d, the same for every way to pair its factors: the
// 1596 entries on and above the diagonal hold only 715 distinct moments of
// degree <= 4, and 55 of y times degree <= 2.  Those 770 sums are all that is
// accumulated.
//
// Eight warps, one program.  Shifting eight of the nine variables cyclically
// (v_j -> v_(j+1 mod 8); the ninth, z = u_dy, stays) maps monomials to
// monomials.  One representative of each orbit, 99 of them, with the variables
// read in an order rotated by the warp's index, and one of the 8 sums without
// any v per warp, cover all 770 from eight warps that run the same
// instructions.  (A program per warp made the warps of an SM evict one
// another's instructions: 2.9 of 7 stalls per issue were fetches.  Nine warps
// and nine cyclic variables take 88 sums, but load the four schedulers
// unevenly, and only 96 registers fit.)  The representatives are products of a
// row term (w v_0 v_k, k <= 3, and the lower degrees) and one of 16 column
// pairs v_c v_d, chosen so that the pairs reach every orbit.
//
// Layout of the work: a CTA of 256 threads takes 16 pixels of one frame (16 x 1
// or 8 x 2).  A lane is a (pixel, half) pair: the two halves of a warp take
// alternate neighbours of the same 16 pixels.  The warps first fill a table of
// (v, z, w z^k, w y z^k) for a segment of neighbour pairs, [pair][entry][lane], then each
// walks it with its 100 sums in registers; no sum crosses a lane until the two
// halves are added.  Partial sums of at most 128 pairs are flushed into shared
// memory, so long windows do not lengthen the FP32 sums.
//
// The solve keeps the matrix in shared memory, [element][pixel]: a lane works
// on its own pixel, so every step of the blocked Cholesky (8 block columns of
// 7, left-looking, one tile per warp, its columns split over the halves) runs
// all its lanes, and operands are read without bank conflicts.  Two CTAs per SM: one
// solves (latency-bound) while the other accumulates (FMA-bound).
//
// Measured at 512 x 512 x 16, 7 x 7 x 3 window: 55.7 ms, against 92.0 ms with the
// Gram accumulated as 36 7 x 7 register tiles (1764 sums per neighbour) and
// factored in registers, 36 threads per pixel.
#include <stdlib.h>

#include <utility>

#include "esim_ad.h"
#include "internal.h"
#include "ptx.cuh"

namespace esim {
namespace {

constexpr int kNQ = 55;                    // unknowns
constexpr int kNA = 56;                    // unknowns + log brightness
constexpr int kPix = 16;                   // pixels per CTA
constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kSums = 100;                 // moments accumulated by a warp
constexpr int kElems = kNA * (kNA + 1) / 2;
constexpr int kPart = 128;                 // neighbour pairs per partial sum
// Table entries of a neighbour: v_0..v_7, v_0..v_6 again, z, w z^0..w z^4, w y z^0..w y z^2.
constexpr int kZ = 15, kWz = 16, kWyz = 21, kEntries = 24;
constexpr int kSegMax = 33, kSegFlush = 16;   // neighbour pairs per table, without and with flushed sums

constexpr float kExp2Scale = 0.84932180028801904272f;  // sqrt(log2(e) / 2)

// Quadratic unknown q (0..44) -> feature pair (a, b), a <= b, a-major order.
__host__ __device__ constexpr int pair_a(int q)
{
    int a = 0;
    while (q >= 9 - a) { q -= 9 - a; ++a; }
    return a;
}
__host__ __device__ constexpr int pair_b(int q)
{
    int a = 0;
    while (q >= 9 - a) { q -= 9 - a; ++a; }
    return a + q;
}

// ------------------------------------------------------- compile-time tables

// A sum in terms of the rotated variables x_0..x_7: row term times x_c x_d (c <=
// d), x_c alone (d = -1), or the warp's own sum without any x (c = -1).
// Row terms: factors x_0 x_k or x_0 or none, times a power of z, times w or w y.
struct Row {
    signed char n, k, z, y;   // number of x factors; the second is x_k; power of z; times y
};
constexpr int kRows = 12;
constexpr Row kRow[kRows] = {{2, 0, 0, 0}, {2, 1, 0, 0}, {2, 2, 0, 0}, {2, 3, 0, 0}, {1, 0, 0, 0}, {1, 0, 1, 0},
                             {0, 0, 0, 0}, {0, 0, 1, 0}, {0, 0, 2, 0}, {0, 0, 3, 0}, {0, 0, 0, 1}, {0, 0, 1, 1}};

struct Sum {
    signed char row, c, d;
};

struct SumList {
    Sum s[kSums];
    int n;
};

// Column pairs, found by a search over hitting sets: every orbit of degree 4
// has a rotation {0, k, c, d} with k <= 3 and (c, d) among them, every orbit of
// degree 3 one {0, c, d}, every orbit of degree 2 one (c, d).
constexpr int kCols = 16;
constexpr signed char kCol[kCols][2] = {{0, 0}, {0, 4}, {0, 5}, {0, 6}, {1, 1}, {1, 2}, {1, 6}, {3, 5},
                                        {3, 7}, {4, 4}, {4, 6}, {4, 7}, {5, 5}, {5, 6}, {6, 6}, {7, 7}};

// The orbit of {v_0..v_(n-1)}: its smallest rotation, as a number.
__host__ __device__ constexpr int orbit(const int (&v)[4], int n)
{
    int best = 1 << 30;
    for (int r = 0; r < 8; ++r) {
        int cnt[8] = {};
        for (int i = 0; i < n; ++i) ++cnt[(v[i] + r) % 8];
        int code = 0;
        for (int k = 0; k < 8; ++k) code = 5 * code + cnt[k];
        if (code < best) best = code;
    }
    return best;
}

__host__ __device__ constexpr SumList sum_list()
{
    SumList l{};
    int seen[kSums] = {}, n_seen = 0;
    for (int q = 0; q < kCols; ++q) {
        const int c = kCol[q][0], d = kCol[q][1];
        for (int row = 0; row <= 6; ++row) {
            if (row == 5) continue;   // goes with row 4
            const int four[4] = {0, row, c, d}, three[4] = {0, c, d, 0}, two[4] = {c, d, 0, 0};
            const int key = row <= 3 ? orbit(four, 4) : row == 4 ? orbit(three, 3) : orbit(two, 2);
            bool dup = false;
            for (int i = 0; i < n_seen; ++i) dup |= seen[i] == key;   // (the codes of different degrees differ)
            if (dup) continue;
            seen[n_seen++] = key;
            auto add = [&](int r) { l.s[l.n++] = Sum{(signed char)r, (signed char)c, (signed char)d}; };
            add(row);
            if (row == 4) add(5);
            if (row == 6) {
                add(7);
                add(8);
                add(10);
            }
        }
    }
    for (int row = 6; row <= 11; ++row) l.s[l.n++] = Sum{(signed char)row, 0, -1};
    l.s[l.n++] = Sum{6, -1, -1};
    return l;
}

constexpr SumList kList = sum_list();
static_assert(kList.n == kSums, "one representative of each orbit");

// Row (= column) of the Gram that holds the product u_p u_q, p <= q, u_0 = 1.
__host__ __device__ constexpr int gram_row(int p, int q)
{
    if (p == 0) return q == 0 ? 54 : 44 + q;
    int z = 0;
    for (int k = 1; k < p; ++k) z += 10 - k;
    return z + (q - p);
}

// First element of tile (I, J), I <= J, of the packed upper triangle: 7 x 7
// tiles in row order, diagonal tiles packed to 28.
__host__ __device__ constexpr int tile_base(int I, int J)
{
    return 28 * I + 49 * (7 * I - I * (I - 1) / 2) + (J > I ? 28 + 49 * (J - I - 1) : 0);
}
static_assert(tile_base(7, 7) + 28 == kElems, "packed triangle");

__host__ __device__ constexpr int diag_elem(int r, int c) { return r * 7 - r * (r - 1) / 2 + (c - r); }

__host__ __device__ constexpr int elem(int i, int j)
{
    const int lo = i < j ? i : j, hi = i < j ? j : i;
    const int I = lo / 7, J = hi / 7;
    return tile_base(I, J) + (I == J ? diag_elem(lo % 7, hi % 7) : (lo % 7) * 7 + hi % 7);
}

// Places of the Gram (element numbers of the packed triangle) that sum i of
// warp w stands for: up to three pairings of its factors, filled up to three
// with the place of y^2, which nothing reads.  Orbits shorter than eight meet
// again in another warp: the first that names a place has it.
struct Places {
    unsigned short e[kSums][kWarps][4];
};

__host__ __device__ constexpr Places places()
{
    Places t{};
    bool taken[kElems] = {};
    const int unread = elem(55, 55);
    for (int i = 0; i < kSums; ++i)
        for (int w = 0; w < kWarps; ++w) {
            // factors as homogeneous indices: 0 the constant 1, 1 v_0 = u_dx, 2 z = u_dy, 3.. v_1..
            const Sum m = kList.s[i];
            const Row r = kRow[m.row];
            int f[4] = {0, 0, 0, 0}, n = 0, z = r.z, y = r.y;
            if (m.c < 0) {   // the warp's own: w z^0..z^4, w y z^0..z^2
                z = w < 5 ? w : w - 5;
                y = w < 5 ? 0 : 1;
            }
            const int x[4] = {0, r.k, m.c, m.d};
            for (int k = 0; k < 4; ++k) {
                const bool used = k < 2 ? k < r.n : x[k] >= 0;
                if (!used) continue;
                const int v = (x[k] + w) % 8;
                f[n++] = v == 0 ? 1 : 2 + v;
            }
            for (int k = 0; k < z; ++k) f[n++] = 2;
            for (int a = 0; a < 4; ++a)
                for (int b = a + 1; b < 4; ++b)
                    if (f[b] < f[a]) {
                        const int h = f[a];
                        f[a] = f[b];
                        f[b] = h;
                    }
            const int at[3] = {y ? elem(gram_row(f[2], f[3]), 55) : elem(gram_row(f[0], f[1]), gram_row(f[2], f[3])),
                               y ? unread : elem(gram_row(f[0], f[2]), gram_row(f[1], f[3])),
                               y ? unread : elem(gram_row(f[0], f[3]), gram_row(f[1], f[2]))};
            for (int k = 0; k < 3; ++k) {
                t.e[i][w][k] = (unsigned short)(taken[at[k]] ? unread : at[k]);
                taken[at[k]] = true;
            }
        }
    return t;
}

__constant__ Places kPlaces = places();

// ------------------------------------------------------------------ the kernel

struct W2Params {
    int W, H, F, r, T, rgb, tiles_x;
    int tw, gx, gy;          // pixel group tw x (16 / tw), groups across and down
    int part;                // neighbour pairs per partial sum
    int flush;               // some window has more pairs than that
    int seg;                 // neighbour pairs per table
    float h, log_eps, ridge;
    const float* radiance;   // [F][C][H][W]
    const float* features;   // [F][7][H][W]
    const float* bandwidth;  // [7]
    float4* packed;          // [F][2][H][W]: (y, normal xyz), (depth, albedo rgb)
    float* alpha;            // [F][H][W]
};

// Dynamic shared memory.  Accumulation: flushed sums [sum][warp][pixel], table
// [pair][entry][lane]; solve: the matrix, over both.
constexpr int kFlushBytes = kSums * kWarps * kPix * 4;
constexpr int kPairBytes = kEntries * 32 * 4;
constexpr int kMatBytes = kElems * kPix * 4;
static_assert(kSegMax * kPairBytes <= kMatBytes && kFlushBytes + kSegFlush * kPairBytes <= kMatBytes,
              "two CTAs per SM");

__global__ void __launch_bounds__(kTilePix) wlr2_pack_kernel(W2Params p)
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
    float4* out = p.packed + (size_t)f * 2 * N;
    out[i] = make_float4(logf(Y + p.log_eps), ft[i], ft[N + i], ft[2 * N + i]);
    out[N + i] = make_float4(ft[3 * N + i], ft[4 * N + i], ft[5 * N + i], ft[6 * N + i]);
}

// One neighbour: x the rotated variables, own the warp's own term.
template <int... I>
__device__ __forceinline__ void add_sums(float (&acc)[kSums], float w, float wy, float z, float own,
                                         const float (&x)[8], std::integer_sequence<int, I...>)
{
    const float wx = w * x[0], wz = w * z, wzz = wz * z;
    const float row[kRows] = {wx * x[0], wx * x[1], wx * x[2], wx * x[3], wx, wz * x[0],
                              w, wz, wzz, wzz * z, wy, wy * z};
    auto term = [&](auto idx, float& a) {
        constexpr Sum m = kList.s[decltype(idx)::value];
        if constexpr (m.c < 0) a += own;
        else if constexpr (m.d < 0) a = fmaf(row[m.row], x[m.c], a);
        else a = fmaf(row[m.row], x[m.c] * x[m.d], a);
    };
    (term(std::integral_constant<int, I>{}, acc[I]), ...);
}

__global__ void __launch_bounds__(kThreads, 2) wlr2_kernel(const W2Params p)
{
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ float s_sf[7];                  // feature scales
    __shared__ float s_c[7][kPix];             // the pixels' features
    __shared__ float s_s2[kNQ];                // squared natural-unit scale of each unknown
    __shared__ float s_d[kNA][kPix];           // equilibration scales
    __shared__ float s_inv[7][kPix];           // 1 / diagonal of U_JJ

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int pi = lane & 15, half = lane >> 4;
    const size_t N = (size_t)p.W * p.H;
    const unsigned gxy = (unsigned)p.gx * (unsigned)p.gy;
    const int f = (int)(blockIdx.x / gxy);
    const int gy = (int)((blockIdx.x % gxy) / (unsigned)p.gx), gx = (int)((blockIdx.x % gxy) % (unsigned)p.gx);
    const int px = gx * p.tw + pi % p.tw, py = gy * (kPix / p.tw) + pi / p.tw;

    if (tid < 7) s_sf[tid] = kExp2Scale / (p.h * p.bandwidth[tid]);
    if (tid < 7 * kPix) {
        // pixels past the image's edge take the group's first: their results are dropped
        const int k = tid >> 4;
        const bool in = px < p.W && py < p.H;
        const size_t ci = in ? (size_t)py * p.W + px : (size_t)gy * (kPix / p.tw) * p.W + (size_t)gx * p.tw;
        const float* rec = reinterpret_cast<const float*>(p.packed + ((size_t)f * 2 + (k < 3 ? 0 : 1)) * N + ci);
        s_c[k][pi] = rec[k < 3 ? 1 + k : k - 3];
    }
    __syncthreads();
    if (tid < kNQ) {
        const float sc = kExp2Scale / p.h;
        auto sdim = [&](int a) { return a < 2 ? sc : s_sf[a - 2]; };
        float s2 = 0.0f;
        if (tid < 45) {
            const float v = sdim(pair_a(tid)) * sdim(pair_b(tid));
            s2 = v * v;
        } else if (tid < 54) {
            const float v = sdim(tid - 45);
            s2 = v * v;
        }
        s_s2[tid] = s2;
    }

    // ---- accumulation: the window's neighbours in pairs, frame by frame
    const int side = 2 * p.r + 1, nq = side * side, npair = (nq + 1) / 2;
    const int tau0 = max(0, f - p.T + 1);
    const int total = npair * (f - tau0 + 1);
    const float s_px = kExp2Scale / (p.h * (float)p.r);
    float* flushed = reinterpret_cast<float*>(sm) + warp * kPix + pi;           // of this warp and pixel, per sum
    float* table = reinterpret_cast<float*>(sm + (p.flush ? kFlushBytes : 0)) + lane;
    float acc[kSums];
#pragma unroll
    for (int i = 0; i < kSums; ++i) acc[i] = 0.0f;
    int run = 0;             // pairs in the registers' partial sums
    bool any = false;        // partial sums have been flushed
    auto flush = [&]() {     // add the halves, then to the flushed sums
#pragma unroll
        for (int i = 0; i < kSums; ++i) {
            const float v = acc[i] + __shfl_xor_sync(0xffffffffu, acc[i], 16);
            float* at = flushed + i * (kWarps * kPix);
            if (half == 0) *at = any ? *at + v : v;
            acc[i] = 0.0f;
        }
        any = true;
        run = 0;
    };
    for (int n0 = 0; n0 < total; n0 += p.seg) {
        const int n = min(p.seg, total - n0);
        for (int i = warp; i < n; i += kWarps) {
            const int k = (n0 + i) / npair, q = 2 * (n0 + i - k * npair) + half;
            const int oy = q / side - p.r, ox = q - (oy + p.r) * side - p.r;
            const int nx = px + ox, ny = py + oy;
            float* e = table + i * (kEntries * 32);
            float a[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            const bool ok = q < nq && nx >= 0 && nx < p.W && ny >= 0 && ny < p.H;
            if (ok) {
                const float4* g = p.packed + (size_t)(tau0 + k) * 2 * N + (size_t)ny * p.W + nx;
                const float4 h0 = __ldg(g), h1 = __ldg(g + N);
                a[0] = h0.x; a[1] = h0.y; a[2] = h0.z; a[3] = h0.w;
                a[4] = h1.x; a[5] = h1.y; a[6] = h1.z; a[7] = h1.w;
            }
            // feature differences are taken before scaling: exact where features are close
            const float u0 = (float)ox * s_px, z = (float)oy * s_px;
            float en = fmaf(u0, u0, z * z);
            e[0] = u0;
            e[8 * 32] = u0;
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                const float u = ok ? (a[1 + j] - s_c[j][pi]) * s_sf[j] : 0.0f;
                en = fmaf(u, u, en);
                e[(1 + j) * 32] = u;
                if (j < 6) e[(9 + j) * 32] = u;
            }
            e[kZ * 32] = z;
            float w = ok ? ex2_approx(-en) : 0.0f, wy = w * a[0];
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                e[(kWz + j) * 32] = w;
                w *= z;
                if (j < 3) {
                    e[(kWyz + j) * 32] = wy;
                    wy *= z;
                }
            }
        }
        __syncthreads();
        for (int j = 0; j < n;) {
            if (p.flush && run == p.part) flush();
            const int m = p.flush ? min(n - j, p.part - run) : n;
            const float* e = table + j * (kEntries * 32);
            const float* ex = e + warp * 32;
#pragma unroll 1
            for (int i = 0; i < m; ++i) {
                const float x[8] = {ex[0], ex[32], ex[64], ex[96], ex[128], ex[160], ex[192], ex[224]};
                add_sums(acc, e[kWz * 32], e[kWyz * 32], e[kZ * 32], ex[kWz * 32], x,
                         std::make_integer_sequence<int, kSums>{});
                e += kEntries * 32;
                ex += kEntries * 32;
            }
            run += m;
            j += m;
        }
        __syncthreads();   // the table is free again
    }
#pragma unroll
    for (int i = 0; i < kSums; ++i) {
        acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
        if (any) acc[i] += flushed[i * (kWarps * kPix)];
    }
    if (p.flush) __syncthreads();   // the matrix takes the place of the flushed sums

    float* mat = reinterpret_cast<float*>(sm) + pi;   // element e of this lane's pixel: mat[e * kPix]
#pragma unroll
    for (int i = 0; i < kSums; ++i) {
        const unsigned short* at = kPlaces.e[i][warp];
#pragma unroll
        for (int k = 0; k < 3; ++k) mat[at[k] * kPix] = acc[i];
    }
    __syncthreads();

    // ---- ridge and Jacobi equilibration scales, A_ab / sqrt(A_aa A_bb) (the
    // log-brightness row keeps scale 1; its own square is never used)
    const float lw = p.ridge * mat[elem(54, 54) * kPix];
    for (int z = tid >> 4; z < kNA; z += kThreads / kPix) {
        if (z == 55) {
            s_d[z][pi] = 1.0f;
            mat[elem(55, 55) * kPix] = 1.0f;
        } else {
            const int J = z / 7, r = z - 7 * J;
            float* at = mat + (tile_base(J, J) + diag_elem(r, r)) * kPix;
            const float a = z < 54 ? fmaf(lw, s_s2[z], *at) : *at;
            // lw is read by every warp: the intercept's entry stays as it is
            if (z < 54) *at = a;
            s_d[z][pi] = rsqrtf(a);
        }
    }
    __syncthreads();

    // ---- left-looking blocked Cholesky A = U^T U over 8 block columns of 7:
    // in step J warp k forms tile (J, J + k) as A - sum_K U_KJ^T U_KL, warp 0
    // factors the diagonal tile, the others solve theirs against it.  A lane
    // holds 4 of its tile's columns: 0-3 in the first half, 3-6 in the second
    // (an odd distance, so that the halves read different banks; column 3 is
    // formed twice).
    const int c0 = 3 * half;
#pragma unroll 1
    for (int J = 0; J < 8; ++J) {
        const int L = J + warp;
        float x[7][4];
        if (L < 8) {
            const bool diag = L == J;
            {
                float dc[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) dc[k] = s_d[7 * L + c0 + k][pi];
                const float* A = mat + tile_base(J, L) * kPix;
#pragma unroll
                for (int i = 0; i < 7; ++i) {
                    const float dr = s_d[7 * J + i][pi];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int c = c0 + k;
                        const int e = diag ? diag_elem(min(i, c), max(i, c)) : i * 7 + c;
                        x[i][k] = A[e * kPix] * (dr * dc[k]);
                    }
                }
            }
#pragma unroll 1
            for (int K = 0; K < J; ++K) {
                const float* UI = mat + tile_base(K, J) * kPix;
                const float* UL = mat + (tile_base(K, L) + c0) * kPix;
#pragma unroll
                for (int m = 0; m < 7; ++m) {
                    float a[7], b[4];
#pragma unroll
                    for (int i = 0; i < 7; ++i) a[i] = UI[(7 * m + i) * kPix];
#pragma unroll
                    for (int k = 0; k < 4; ++k) b[k] = UL[(7 * m + k) * kPix];
#pragma unroll
                    for (int i = 0; i < 7; ++i)
#pragma unroll
                        for (int k = 0; k < 4; ++k) x[i][k] = fmaf(-a[i], b[k], x[i][k]);
                }
            }
            if (diag) {
                float* D = mat + tile_base(J, J) * kPix;
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 7; ++i)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (i <= c0 + k) D[diag_elem(i, c0 + k) * kPix] = x[i][k];
                __syncwarp();
                float g[28];
#pragma unroll
                for (int e = 0; e < 28; ++e) g[e] = D[e * kPix];
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 7; ++i) {
                    const float piv = sqrtf(fmaxf(g[diag_elem(i, i)], 1e-30f));
                    const float inv = 1.0f / piv;
                    g[diag_elem(i, i)] = piv;
#pragma unroll
                    for (int k = i + 1; k < 7; ++k) g[diag_elem(i, k)] *= inv;
#pragma unroll
                    for (int m = i + 1; m < 7; ++m)
#pragma unroll
                        for (int k = m; k < 7; ++k)
                            g[diag_elem(m, k)] = fmaf(-g[diag_elem(i, m)], g[diag_elem(i, k)], g[diag_elem(m, k)]);
                    s_inv[i][pi] = inv;
                }
#pragma unroll
                for (int e = 0; e < 28; ++e) D[e * kPix] = g[e];
                // With the intercept last and y appended, U[54][55] = (U^-T b)_54 and
                // theta_54 = U[54][55] / U[54][54] in the equilibrated basis.
                if (J == 7 && half == 0 && px < p.W && py < p.H)
                    p.alpha[(size_t)f * N + (size_t)py * p.W + px] =
                        g[diag_elem(5, 6)] / g[diag_elem(5, 5)] * s_d[54][pi];
            }
        }
        __syncthreads();
        if (L < 8 && L > J) {
            const float* D = mat + tile_base(J, J) * kPix;
            float* X = mat + (tile_base(J, L) + c0) * kPix;
#pragma unroll
            for (int i = 0; i < 7; ++i) {
                const float inv = s_inv[i][pi];
#pragma unroll
                for (int m = 0; m < i; ++m) {
                    const float um = D[diag_elem(m, i) * kPix];
#pragma unroll
                    for (int k = 0; k < 4; ++k) x[i][k] = fmaf(-um, x[m][k], x[i][k]);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) x[i][k] *= inv;
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 7; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) X[(7 * i + k) * kPix] = x[i][k];
        }
        __syncthreads();
    }
}

bool desc_ok(const esim_ad_wlr_desc* d)
{
    return d && d->struct_size == sizeof(esim_ad_wlr_desc) && d->width >= 1 && d->height >= 1 &&
           d->sequence >= 1 && d->radius >= 1 && d->radius <= kMaxRadius && d->frames >= 1 &&
           d->frames <= kMaxFrames && (d->radiance_fmt == ESIM_AD_LUMA_F32 || d->radiance_fmt == ESIM_AD_RGB_F32) &&
           d->h > 0.0f && d->ridge > 0.0f && d->log_eps >= 0.0f;
}

// Neighbour pairs per partial sum: kPart, or, with ESIM_AD_WLR2_GROUPS = g (2,
// 4 or 8), few enough to cut a window of `pairs` pairs into g partial sums.
int part_pairs(int pairs)
{
    if (const char* e = getenv("ESIM_AD_WLR2_GROUPS")) {
        const int g = atoi(e);
        if (g == 2 || g == 4 || g == 8) return pairs / g < 1 ? 1 : pairs / g < kPart ? pairs / g : kPart;
    }
    return kPart;
}

}  // namespace
}  // namespace esim

using namespace esim;

extern "C" size_t esim_ad_wlr2_workspace_size(const esim_ad_wlr_desc* d)
{
    if (!desc_ok(d)) return 0;
    return (size_t)d->sequence * 2 * (size_t)d->width * d->height * sizeof(float4);
}

extern "C" esim_ad_status esim_ad_wlr2_forward(const esim_ad_wlr_desc* d, const float* radiance,
                                               const float* features, const float* bandwidth, float* alpha,
                                               void* workspace, void* cuda_stream)
{
    if (!desc_ok(d) || !radiance || !features || !bandwidth || !alpha || !workspace) return ESIM_AD_EINVAL;
    W2Params p;
    p.W = d->width;
    p.H = d->height;
    p.F = d->sequence;
    p.r = d->radius;
    p.T = d->frames;
    p.rgb = d->radiance_fmt == ESIM_AD_RGB_F32 ? 1 : 0;
    p.tiles_x = (d->width + kTileX - 1) / kTileX;
    p.h = d->h;
    p.log_eps = d->log_eps;
    p.ridge = d->ridge;
    p.radiance = radiance;
    p.features = features;
    p.bandwidth = bandwidth;
    p.packed = static_cast<float4*>(workspace);
    p.alpha = alpha;
    if (d->sequence > 65535) return ESIM_AD_EINVAL;   // frames index the pack grid's y dimension
    // pixel groups 16 x 1, or 8 x 2 where that takes fewer
    auto groups = [&](int tw) {
        return (unsigned long long)((p.W + tw - 1) / tw) * ((p.H + kPix / tw - 1) / (kPix / tw));
    };
    p.tw = groups(8) < groups(16) ? 8 : 16;
    p.gx = (p.W + p.tw - 1) / p.tw;
    p.gy = (p.H + kPix / p.tw - 1) / (kPix / p.tw);
    const unsigned long long n = groups(p.tw) * (unsigned long long)p.F;
    if (n > 0x7fffffffull) return ESIM_AD_EINVAL;
    const int S = 2 * d->radius + 1;
    const int pairs = (S * S + 1) / 2 * (d->frames < d->sequence ? d->frames : d->sequence);
    p.part = part_pairs(pairs);
    p.flush = pairs > p.part ? 1 : 0;
    // tables of equal length, as many pairs as fit beside what else is kept
    const int cap = p.flush ? kSegFlush : kSegMax, segs = (pairs + cap - 1) / cap;
    p.seg = (pairs + segs - 1) / segs;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const dim3 pack_grid(p.tiles_x * ((d->height + kTileY - 1) / kTileY), d->sequence);
    wlr2_pack_kernel<<<pack_grid, kTilePix, 0, s>>>(p);
    if (cudaGetLastError() != cudaSuccess) return ESIM_AD_ECUDA;
    if (cudaFuncSetAttribute(wlr2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMatBytes) != cudaSuccess)
        return ESIM_AD_ECUDA;
    wlr2_kernel<<<(unsigned)n, kThreads, kMatBytes, s>>>(p);
    return cudaGetLastError() == cudaSuccess ? ESIM_AD_OK : ESIM_AD_ECUDA;
}
