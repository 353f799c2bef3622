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
// row term (w v_0 v_k, and the lower degrees) and one of 16 column pairs v_c
// v_d, chosen so that the pairs reach every orbit and that the rows that a
// column needs come in twos: 98 of the 100 sums are updated by 49 packed FMAs.
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
// on its own pixel, so every step of the blocked Cholesky (7 block columns of
// 8, one tile per warp, its even and odd columns on the halves) runs all its
// lanes, and operands are read without bank conflicts.  Two CTAs per SM: one
// solves (latency-bound) while the other accumulates (FMA-bound).  Over both
// phases the FMA pipe is 41% busy and half of the issue slots are used; the first
// stall is the barriers of the solve and of the table.
//
// Measured at 512 x 512 x 16, 7 x 7 x 3 window: 46.7 ms (55.7 with single FMAs,
// blocks of 7 and a wholly left-looking order), against 92.0 ms with the
// Gram accumulated as 36 7 x 7 register tiles (1764 sums per neighbour) and
// factored in registers, 36 threads per pixel.  Small inputs stay with that one
// (wlr2_gram.cu).
#include <stdlib.h>

#include <utility>

#include "esim_ad.h"
#include "internal.h"
#include "ptx.cuh"
#include "wlr2.cuh"

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

// ------------------------------------------------------- compile-time tables

// A sum in terms of the rotated variables x_0..x_7: row term times x_c x_d (c <=
// d), x_c alone (d = -1), or the warp's own sum without any x (c = -1).
// Row terms: factors x_0 x_k or x_0 or none, times a power of z, times w or w y;
// rows 2r and 2r + 1 are a pair.
struct Row {
    signed char n, k, z, y;   // number of x factors; the second is x_k; power of z; times y
};
constexpr int kRows = 12;
constexpr Row kRow[kRows] = {{2, 0, 0, 0}, {2, 2, 0, 0}, {2, 1, 0, 0}, {2, 4, 0, 0}, {1, 0, 0, 0}, {1, 0, 1, 0},
                             {0, 0, 0, 0}, {0, 0, 1, 0}, {0, 0, 2, 0}, {0, 0, 0, 1}, {0, 0, 3, 0}, {0, 0, 1, 1}};

struct Sum {
    signed char row, c, d;
};

struct SumList {
    Sum s[kSums];   // 2i and 2i + 1: a pair of rows times one column, but for the last two
    int n;
};

// Column pairs in the order of their use, found by a search: every orbit of
// degree 4 has a rotation {0, k, c, d}, k in {0, 1, 2, 4}, with (c, d) among
// them, every orbit of degree 3 one {0, c, d}, every orbit of degree 2 one
// (c, d); and taken in this order 42 of the 43 orbits of degree 4 fall into
// whole row pairs.
constexpr int kCols = 16;
constexpr signed char kCol[kCols][2] = {{7, 7}, {0, 6}, {1, 7}, {5, 5}, {1, 5}, {0, 7}, {0, 3}, {5, 6},
                                        {0, 0}, {2, 6}, {6, 6}, {5, 7}, {3, 6}, {0, 4}, {1, 4}, {0, 5}};

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
    int seen[kSums] = {}, n_seen = 0;   // orbits (the codes of different degrees differ)
    Sum last{};                         // the single sum of degree 4
    auto is_new = [&](int key) {
        for (int i = 0; i < n_seen; ++i)
            if (seen[i] == key) return false;
        return true;
    };
    for (int q = 0; q < kCols; ++q) {
        const int c = kCol[q][0], d = kCol[q][1];
        auto add = [&](int row, int cc, int dd) { l.s[l.n++] = Sum{(signed char)row, (signed char)cc, (signed char)dd}; };
        for (int r = 0; r < 2; ++r) {
            const int lo[4] = {0, kRow[2 * r].k, c, d}, hi[4] = {0, kRow[2 * r + 1].k, c, d};
            const int kl = orbit(lo, 4), kh = orbit(hi, 4);
            if (is_new(kl) && is_new(kh) && kl != kh) {
                seen[n_seen++] = kl;
                seen[n_seen++] = kh;
                add(2 * r, c, d);
                add(2 * r + 1, c, d);
            }
        }
        for (int row = 0; row < 4; ++row) {
            const int four[4] = {0, kRow[row].k, c, d}, key = orbit(four, 4);
            if (is_new(key)) {
                seen[n_seen++] = key;
                last = Sum{(signed char)row, (signed char)c, (signed char)d};
            }
        }
        const int three[4] = {0, c, d, 0}, two[4] = {c, d, 0, 0};
        if (is_new(orbit(three, 3))) {
            seen[n_seen++] = orbit(three, 3);
            add(4, c, d);
            add(5, c, d);
        }
        if (is_new(orbit(two, 2))) {
            seen[n_seen++] = orbit(two, 2);
            for (int row = 6; row < 10; ++row) add(row, c, d);
        }
    }
    for (int row = 6; row < 12; ++row) l.s[l.n++] = Sum{(signed char)row, 0, -1};
    l.s[l.n++] = last;
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

// First element of tile (I, J), I <= J, of the packed upper triangle: 8 x 8
// tiles in row order, diagonal tiles packed to 36.
constexpr int kB = 8, kNB = kNA / kB, kDiag = kB * (kB + 1) / 2;
__host__ __device__ constexpr int tile_base(int I, int J)
{
    return kDiag * I + kB * kB * ((kNB - 1) * I - I * (I - 1) / 2) + (J > I ? kDiag + kB * kB * (J - I - 1) : 0);
}
static_assert(tile_base(kNB - 1, kNB - 1) + kDiag == kElems, "packed triangle");

__host__ __device__ constexpr int diag_elem(int r, int c) { return r * kB - r * (r - 1) / 2 + (c - r); }

__host__ __device__ constexpr int elem(int i, int j)
{
    const int lo = i < j ? i : j, hi = i < j ? j : i;
    const int I = lo / kB, J = hi / kB;
    return tile_base(I, J) + (I == J ? diag_elem(lo % kB, hi % kB) : (lo % kB) * kB + hi % kB);
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
__device__ __forceinline__ void add_sums(float2 (&acc)[kSums / 2], float w, float wy, float z, float own,
                                         const float (&x)[8], std::integer_sequence<int, I...>)
{
    const float wx = w * x[0], wz = w * z, wzz = wz * z;
    const float2 row[kRows / 2] = {make_float2(wx * x[0], wx * x[2]), make_float2(wx * x[1], wx * x[4]),
                                   make_float2(wx, wz * x[0]),        make_float2(w, wz),
                                   make_float2(wzz, wy),              make_float2(wzz * z, wy * z)};
    auto term = [&](auto idx, float2& a) {
        constexpr int i = decltype(idx)::value;
        constexpr Sum m = kList.s[2 * i];
        if constexpr (2 * i + 2 == kSums) {
            a.x = fmaf(m.row & 1 ? row[m.row / 2].y : row[m.row / 2].x, x[m.c] * x[m.d], a.x);
            a.y += own;
        } else {
            float p = x[m.c];
            if constexpr (m.d >= 0) p *= x[m.d];
            a = __ffma2_rn(row[m.row / 2], make_float2(p, p), a);
        }
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
    __shared__ float s_inv[kB][kPix];           // 1 / diagonal of U_JJ

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
    float2 acc[kSums / 2];
#pragma unroll
    for (int i = 0; i < kSums / 2; ++i) acc[i] = make_float2(0.0f, 0.0f);
    int run = 0;             // pairs in the registers' partial sums
    bool any = false;        // partial sums have been flushed
    auto both_halves = [&](float v) { return v + __shfl_xor_sync(0xffffffffu, v, 16); };
    auto flush = [&]() {
#pragma unroll
        for (int i = 0; i < kSums / 2; ++i) {
            const float v[2] = {both_halves(acc[i].x), both_halves(acc[i].y)};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float* at = flushed + (2 * i + h) * (kWarps * kPix);
                if (half == 0) *at = any ? *at + v[h] : v[h];
            }
            acc[i] = make_float2(0.0f, 0.0f);
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
                         std::make_integer_sequence<int, kSums / 2>{});
                e += kEntries * 32;
                ex += kEntries * 32;
            }
            run += m;
            j += m;
        }
        __syncthreads();   // the table is free again
    }
#pragma unroll
    for (int i = 0; i < kSums / 2; ++i) {
        acc[i] = make_float2(both_halves(acc[i].x), both_halves(acc[i].y));
        if (any) {
            acc[i].x += flushed[2 * i * (kWarps * kPix)];
            acc[i].y += flushed[(2 * i + 1) * (kWarps * kPix)];
        }
    }
    if (p.flush) __syncthreads();   // the matrix takes the place of the flushed sums

    float* mat = reinterpret_cast<float*>(sm) + pi;   // element e of this lane's pixel: mat[e * kPix]
#pragma unroll
    for (int i = 0; i < kSums; ++i) {
        const unsigned short* at = kPlaces.e[i][warp];
#pragma unroll
        for (int k = 0; k < 3; ++k) mat[at[k] * kPix] = i & 1 ? acc[i / 2].y : acc[i / 2].x;
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
            float* at = mat + elem(z, z) * kPix;
            const float a = z < 54 ? fmaf(lw, s_s2[z], *at) : *at;
            // lw is read by every warp: the intercept's entry stays as it is
            if (z < 54) *at = a;
            s_d[z][pi] = rsqrtf(a);
        }
    }
    __syncthreads();

    // ---- blocked Cholesky A = U^T U over 7 block columns of 8.  A warp forms one
    // tile (I, L) as A - sum_K U_KI^T U_KL; a lane holds 4 of its columns, the
    // even ones in the first half and the odd ones in the second (neighbouring
    // elements lie in different banks).  Left-looking over block columns 0-3,
    // then their part of the last six tiles at once (six warps, where the
    // left-looking order would leave it to three, two and one), then
    // left-looking over the rest.
    constexpr int kSplit = 4;
    float x[kB][4];
    auto form = [&](int I, int L, int K0, int K1, bool scale) {
        const float* A = mat + tile_base(I, L) * kPix;
        float2 v[kB][2];
        float dc[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) dc[k] = scale ? -s_d[kB * L + 2 * k + half][pi] : -1.0f;
#pragma unroll
        for (int i = 0; i < kB; ++i) {
            const float dr = scale ? s_d[kB * I + i][pi] : 1.0f;
            float a[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int c = 2 * k + half;
                const int e = I == L ? diag_elem(min(i, c), max(i, c)) : i * kB + c;
                a[k] = A[e * kPix] * (dr * dc[k]);
            }
            v[i][0] = make_float2(a[0], a[1]);
            v[i][1] = make_float2(a[2], a[3]);
        }
#pragma unroll 1
        for (int K = K0; K < K1; ++K) {
            const float* UI = mat + tile_base(K, I) * kPix;
            const float* UL = mat + (tile_base(K, L) + half) * kPix;
#pragma unroll
            for (int m = 0; m < kB; ++m) {
                const float2 b0 = make_float2(UL[kB * m * kPix], UL[(kB * m + 2) * kPix]);
                const float2 b1 = make_float2(UL[(kB * m + 4) * kPix], UL[(kB * m + 6) * kPix]);
#pragma unroll
                for (int i = 0; i < kB; ++i) {
                    const float a = UI[(kB * m + i) * kPix];
                    v[i][0] = __ffma2_rn(make_float2(a, a), b0, v[i][0]);
                    v[i][1] = __ffma2_rn(make_float2(a, a), b1, v[i][1]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kB; ++i) {
            x[i][0] = -v[i][0].x;
            x[i][1] = -v[i][0].y;
            x[i][2] = -v[i][1].x;
            x[i][3] = -v[i][1].y;
        }
    };
    auto put = [&](int I, int L) {
        float* A = mat + tile_base(I, L) * kPix;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kB; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int c = 2 * k + half;
                if (I != L) A[(i * kB + c) * kPix] = x[i][k];
                else if (i <= c) A[diag_elem(i, c) * kPix] = x[i][k];
            }
        __syncwarp();
    };
#pragma unroll 1
    for (int J = 0; J < kNB; ++J) {
        if (J == kSplit) {
            if (warp < 6) {
                const int I = warp < 3 ? 4 : warp < 5 ? 5 : 6, L = warp < 3 ? 4 + warp : warp < 5 ? 2 + warp : 6;
                form(I, L, 0, kSplit, true);
                put(I, L);
            }
            __syncthreads();
        }
        const int L = J + warp;
        if (L < kNB) form(J, L, J < kSplit ? 0 : kSplit, J, J < kSplit);
        if (warp == 0) {
            // the diagonal tile, by every lane for its own pixel
            put(J, J);
            float* D = mat + tile_base(J, J) * kPix;
            float g[kDiag];
#pragma unroll
            for (int e = 0; e < kDiag; ++e) g[e] = D[e * kPix];
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kB; ++i) {
                // 1 / sqrt of the pivot: one Newton step on the approximation, within 0.62 units in
                // the last place (a rounded root and division: 0.75)
                const float piv = fmaxf(g[diag_elem(i, i)], 1e-30f), r0 = rsqrtf(piv);
                const float inv = fmaf(0.5f * r0, fmaf(-piv * r0, r0, 1.0f), r0);
#pragma unroll
                for (int k = i + 1; k < kB; ++k) g[diag_elem(i, k)] *= inv;
#pragma unroll
                for (int m = i + 1; m < kB; ++m)
#pragma unroll
                    for (int k = m; k < kB; ++k)
                        g[diag_elem(m, k)] = fmaf(-g[diag_elem(i, m)], g[diag_elem(i, k)], g[diag_elem(m, k)]);
                s_inv[i][pi] = inv;
                // With the intercept last and y appended, U[54][55] = (U^-T b)_54 and
                // theta_54 = U[54][55] / U[54][54] in the equilibrated basis.
                if (i == kB - 2 && J == kNB - 1 && half == 0 && px < p.W && py < p.H)
                    p.alpha[(size_t)f * N + (size_t)py * p.W + px] = g[diag_elem(i, i + 1)] * inv * s_d[54][pi];
            }
#pragma unroll
            for (int e = 0; e < kDiag; ++e) D[e * kPix] = g[e];
        }
        if (J == kNB - 1) break;
        __syncthreads();
        if (L < kNB && L > J) {
            const float* D = mat + tile_base(J, J) * kPix;
#pragma unroll
            for (int i = 0; i < kB; ++i) {
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
            put(J, L);
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

// Inputs of at most this many pixel groups take the Gram kernel (wlr2_gram.cu, with
// both sides measured); ESIM_AD_WLR2_SMALL overrides the line.
unsigned long long small_groups()
{
    if (const char* e = getenv("ESIM_AD_WLR2_SMALL")) {
        if (*e) return strtoull(e, nullptr, 10);
    }
    return 64;
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
    const bool small = n <= small_groups();
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
    if (small) {
        const cudaError_t e = launch_wlr2_gram(p, s);
        return e == cudaSuccess ? ESIM_AD_OK : e == cudaErrorInvalidValue ? ESIM_AD_EINVAL : ESIM_AD_ECUDA;
    }
    if (cudaFuncSetAttribute(wlr2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMatBytes) != cudaSuccess)
        return ESIM_AD_ECUDA;
    wlr2_kernel<<<(unsigned)n, kThreads, kMatBytes, s>>>(p);
    return cudaGetLastError() == cudaSuccess ? ESIM_AD_OK : ESIM_AD_ECUDA;
}
