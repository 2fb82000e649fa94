// Block one-sided Jacobi SVD in FP32 for the charge sectors of the two-site wavefunction
// (the decomposition of Eq. (svd), Sec. II).
//
// The columns of every sector matrix W (p x n, column-major, n <= p) are cut into blocks of 16.
// A sweep pairs every block with every other block once (round-robin ordering of the blocks), one
// pair per CTA: it stages the p x 32 columns in shared memory, forms their 32 x 32 Gram matrix,
// diagonalises it with two-sided cyclic Jacobi, orders the eigenvectors by decreasing eigenvalue
// (block I receives the larger ones), and rotates the staged columns and the matching columns of V
// by that orthogonal matrix.  The sector has converged when a sweep finds no pair to rotate; the
// test of a pair is computed from the current columns, so the inexact inner solve is corrected by
// the next visit.  With the GPU to itself the caller runs all sweeps in one cooperative launch (a
// queue ordered by dependencies); while regions run concurrently, each round is its own launch
// (kernel boundaries order the rounds and nothing spins, so the regions' kernels interleave freely).
//
// What bounds it is a chain: a block's pairs follow each other (nb - 1 of them a sweep, 6 to 8
// sweeps), so the time is rounds x the latency of one task; the FP32 units are mostly idle.  Hence:
// - Pairs within a block are solved once a sweep (31 inner rounds over all 496 pairs); the other
//   visits turn only the 256 pairs across (16 inner rounds).  Inner rounds read one copy of G and
//   write another (one barrier each), rotations are two reciprocal roots, every warp works out all
//   16 of a round.
// - W is published before V is rotated: the next pairs of these blocks wait for W alone.
// - Two CTAs share an SM where the columns allow it: one's barriers hide behind the other's work.
// - A task waits for its own two blocks, not for its sector's previous round.
// Kernel time over a split, before (two inner sweeps of 31 rounds with two barriers, one CTA an SM,
// sector rounds in step) and now: mixed-mode cylinder bond m = 2000 32.0 -> 18.4 ms, chain FP64 m = 512
// 14.8 -> 9.1 ms, accurate m = 1000 19.5 -> 12.8 ms.
//
// A pair of columns (u, v) is rotated when |g_uv| > tol * |w_u| |w_v| + noise * (|w_u| + |w_v|),
// with noise = c * eps_f32 * sigma_max: the second term is the absolute rounding level of FP32
// columns of a matrix whose largest singular value is sigma_max.  Pairs below it are left as
// they are; their effect on the kept weight is below eps_f32 * sigma_max^2.
//
// Unchanged pairs are skipped: every block records the time (sweep * rounds + round + 1) it was
// last rotated, every block pair the time it was last found converged; a pair found converged
// after both of its blocks' last rotations has the same Gram matrix as then (and the noise level
// only grows), so it is converged still and is not staged again.  In a round a block belongs to
// one pair only, so each stamp has one writer per round; they are read after the queue's wait for
// that pair (or the kernel boundary), from L2.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

#include "internal.h"

namespace pd {

namespace {

constexpr int BJ_B = 16;                     // columns per block
constexpr int BJ_K = 2 * BJ_B;               // columns of a block pair (= warp width)
constexpr int BJ_GLD = BJ_K + 1;             // row stride of Gram matrices
constexpr int BJ_QLD = BJ_K + 4;             // row stride of rotations (16-byte aligned rows)
constexpr int BJ_THREADS = 256;
constexpr int BJ_WARPS = BJ_THREADS / 32;
constexpr int BJ_SMEM_SM = 227 * 1024;       // shared memory of an SM (1 KB of it per resident CTA)

struct alignas(16) BjShared {
    union {
        float Gp[BJ_WARPS / 2][BJ_K * BJ_K];   // partial Gram matrices, until they are summed
        float Q[2][BJ_K * BJ_QLD];             // accumulated rotation; its column-permuted copy
    };
    float G[2][BJ_K * BJ_GLD];                 // Gram matrix, one copy read and one written a round
    int gcol[BJ_K];                            // sector column of staged column u (-1: padding)
    int pos[BJ_K];                             // pos[v] = position of eigenvector v
    float gmax;                                // largest squared column norm seen in the sector
    int qitem, qsec, qsweep, qround, qpair, qok;   // work queue: item taken by this CTA, its state
    int cur;                                   // which copy of G holds the inner solve's result
};
static_assert(sizeof(BjShared) % 16 == 0, "staging area must stay 16-byte aligned");

// Staged columns: column-major, X[u * ldx + r].  The stride is 4 mod 32, so four rows of eight columns
// are read without bank conflicts.
__host__ __device__ constexpr int bj_ldx(int rows) { return (rows + 31) / 32 * 32 + 4; }
// Rows that fit when `ctas` CTAs share an SM.
constexpr int bj_fit(int ctas) {
    return ((BJ_SMEM_SM / ctas - 1024 - (int)sizeof(BjShared)) / (BJ_K * 4) - 4) / 32 * 32;
}

__device__ __forceinline__ int rr_pos(int pos, int round, int npad) {
    return pos == 0 ? 0 : ((pos - 1 + round) % (npad - 1)) + 1;
}

__device__ __forceinline__ bool bj_need(float guv, float guu, float gvv, float tol, float noise) {
    if (!(guu > 0.f) || !(gvv > 0.f)) return false;
    const float su = guu * rsqrtf(guu), sv = gvv * rsqrtf(gvv);   // approximate roots: a threshold
    return fabsf(guv) > tol * su * sv + noise * (su + sv);
}

template <int BYTES>
__device__ __forceinline__ void cp_async(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// X[u][r] = src[gcol[u] * ld + r0 + r] for r < rows, zero for padding columns and up to the next
// multiple of four rows, as asynchronous copies (the caller waits).  A warp takes whole columns.
template <int VEC>
__device__ __forceinline__ void bj_stage_vec(float* __restrict__ X, int ldx, const float* __restrict__ src, int ld,
                                             int r0, int rows, const int* __restrict__ gcol) {
    const int lane = threadIdx.x & 31;
    const int whole = rows / VEC * VEC;
#pragma unroll
    for (int i = 0; i < BJ_K / BJ_WARPS; ++i) {
        const int u = (threadIdx.x >> 5) + BJ_WARPS * i, c = gcol[u];
        float* x = X + u * ldx;
        if (c >= 0) {
            const float* col = src + (long long)c * ld + r0;
            for (int r = VEC * lane; r < whole; r += VEC * 32) cp_async<4 * VEC>(x + r, col + r);
            if (VEC > 1 && lane < rows - whole) cp_async<4>(x + whole + lane, col + whole + lane);
            if (lane < ((4 - (rows & 3)) & 3)) x[rows + lane] = 0.f;
        } else {
            for (int r = lane; r < ((rows + 3) & ~3); r += 32) x[r] = 0.f;
        }
    }
}
__device__ __forceinline__ void bj_stage(float* __restrict__ X, int ldx, const float* __restrict__ src, int ld, int r0,
                                         int rows, const int* __restrict__ gcol) {
    // widest copy that every column's start allows
    const unsigned align = (unsigned)(reinterpret_cast<uintptr_t>(src) >> 2) | (unsigned)ld | (unsigned)r0;
    if ((align & 3) == 0) bj_stage_vec<4>(X, ldx, src, ld, r0, rows, gcol);
    else if ((align & 1) == 0) bj_stage_vec<2>(X, ldx, src, ld, r0, rows, gcol);
    else bj_stage_vec<1>(X, ldx, src, ld, r0, rows, gcol);
}

// Gram accumulation over `rows` staged rows: lane l holds the elements (u, v) = (l % 4 + 4 i, l / 4 + 8 j),
// i < 8, j < 4 (neighbouring columns in one load: no bank conflicts); a warp takes every eighth group of
// four rows, 128 FMA on 12 sixteen-byte loads.
__device__ __forceinline__ void bj_gram_acc(float (&acc)[8][4], const float* __restrict__ X, int ldx, int rows) {
    const int lane = threadIdx.x & 31;
    const float* xu = X + (lane & 3) * ldx;
    const float* xv = X + (lane >> 2) * ldx;
    for (int r = 4 * (threadIdx.x >> 5); r < rows; r += 4 * BJ_WARPS) {
        float4 b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(xv + 8 * j * ldx + r);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 a = *reinterpret_cast<const float4*>(xu + 4 * i * ldx + r);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a.x, b[j].x, acc[i][j]);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a.y, b[j].y, acc[i][j]);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a.z, b[j].z, acc[i][j]);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a.w, b[j].w, acc[i][j]);
        }
    }
}
// G[0] = sum of the warps' elements (a fixed order), in two steps to halve the space.
__device__ __forceinline__ void bj_gram_reduce(BjShared& S, const float (&acc)[8][4]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w >= BJ_WARPS / 2) {
        float* gp = S.Gp[w - BJ_WARPS / 2] + lane;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) gp[(4 * i + j) * 32] = acc[i][j];
    }
    __syncthreads();
    if (w < BJ_WARPS / 2) {
        float* gp = S.Gp[w] + lane;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) gp[(4 * i + j) * 32] += acc[i][j];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < BJ_K * BJ_K / BJ_THREADS; ++q) {
        const int e = threadIdx.x + q * BJ_THREADS, ij = e >> 5;
        const int u = (lane & 3) + 4 * (ij >> 2), v = (lane >> 2) + 8 * (ij & 3);
        S.G[0][u * BJ_GLD + v] = (S.Gp[0][e] + S.Gp[1][e]) + (S.Gp[2][e] + S.Gp[3][e]);
    }
    __syncthreads();
}

// dst[gcol[c] * ld + r0 + r] = sum_u X[u][r] Qp[u][c] for c < k: a warp takes 128 rows (four a lane, a
// warp's rows next to each other) and 8 columns, straight to global memory.
__device__ __forceinline__ void bj_rotate_out(const float* __restrict__ X, int ldx, int rows, const float* __restrict__ Qp,
                                              float* __restrict__ dst, int ld, int r0, const int* __restrict__ gcol,
                                              int k) {
    const int lane = threadIdx.x & 31;
    const int items = (rows + 127) / 128 * 4;
    for (int it = threadIdx.x >> 5; it < items; it += BJ_WARPS) {
        const int c0 = 8 * (it & 3), rb = (it >> 2) * 128 + lane;
        if (c0 >= k) continue;
        int ri[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) ri[i] = min(rb + 32 * i, rows - 1);
        float acc[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll 4
        for (int u = 0; u < BJ_K; ++u) {
            const float4 qa = *reinterpret_cast<const float4*>(Qp + u * BJ_QLD + c0);
            const float4 qb = *reinterpret_cast<const float4*>(Qp + u * BJ_QLD + c0 + 4);
            const float q[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float x = X[u * ldx + ri[i]];
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(x, q[j], acc[i][j]);
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (c0 + j >= k) break;
            float* col = dst + (long long)gcol[c0 + j] * ld + r0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (rb + 32 * i < rows) col[rb + 32 * i] = acc[i][j];
        }
    }
}

// Rotation (c, s) annihilating g_pq of the pair (p, q): new_p = c p - s q, new_q = s p + c q.  With
// d = g_qq - g_pp and h = 2 g_pq: cos 2t = |d| / sqrt(d^2 + h^2), c^2 = (1 + cos 2t) / 2, s = h sign(d) /
// (2 c sqrt(d^2 + h^2)) -- a chain of two reciprocal roots (d and h are scaled by a power of two
// first).  The angle may be slightly inexact (approximate roots; the next visit corrects it), but c
// and s are normalised to c^2 + s^2 = 1 within rounding, since the accumulated rotations must stay
// orthogonal.
__device__ __forceinline__ void bj_rot(float gpp, float gqq, float gpq, float& c, float& s) {
    float d = gqq - gpp, h = gpq;
    const float m = fmaxf(fabsf(d), fabsf(h));
    // 2^-exponent(m): its bits are 254 - e in the exponent field; 2^-126 from 2^126 on
    const float sc = __int_as_float(max(0x7f000000 - (__float_as_int(m) & 0x7f800000), 0x00800000));
    d *= sc;
    h *= sc;                                           // (2 sc would overflow where m is not normal)
    h += h;
    const float r = rsqrtf(fmaf(d, d, h * h));
    const float c2 = fmaf(0.5f * fabsf(d), r, 0.5f);
    const float y = rsqrtf(c2);
    c = c2 * y;
    s = (d >= 0.f ? 0.5f : -0.5f) * h * r * y;
    const float f = fmaf(-0.5f, fmaf(s, s, c * c), 1.5f);
    c *= f;
    s *= f;
}

// The rotations of 16 pairs, one a lane (identity where the pair needs none); false: none needs one.
__device__ __forceinline__ bool bj_decide(float gpp, float gqq, float gpq, float tol, float noise, float& c, float& s) {
    bj_rot(gpp, gqq, gpq, c, s);
    // (the test runs beside the rotation's chain; NaN in an unused rotation is dropped here)
    const bool rot = bj_need(gpq, gpp, gqq, tol, noise);
    c = rot ? c : 1.f;
    s = rot ? s : 0.f;
    return __any_sync(0xffffffffu, rot) != 0;
}

// The inner solve: a two-sided Jacobi on the Gram matrix S.G[0], in one of two forms.  It need not be
// exact (each pair's next visit corrects it), but a round is a chain of dependent steps -- read the 16
// pairs, work out their rotations, apply them, barrier -- so the number of rounds and their length are
// what a task's latency is made of.  Every warp works out all 16 rotations itself (lane l and l + 16:
// pair l) and gets the others' by shuffle: one barrier a round.  The result's diagonal is in S.G[S.cur].
constexpr int BJ_SOLVERS = 128;               // threads of the solve proper
template <int N>
__device__ __forceinline__ void bj_sync_some() { asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory"); }

// All 496 pairs, 31 rounds of the round-robin tournament (players' numbers go up by one a round, 1..31
// cyclic, 0 fixed), Q accumulated in S.Q[0].  A thread rotates two 2 x 2 blocks of G (rows of pairs t /
// 16 and t / 16 + 8, columns of pair t % 16; the blocks partition G) from one copy into the other, and
// four column pairs of one row of Q in place.
__device__ __forceinline__ void bj_pair(int rnd, int i, int& lo, int& hi) {
    int a = i + rnd, b = BJ_K - 1 - i + rnd;
    a = i == 0 ? 0 : (a > BJ_K - 1 ? a - (BJ_K - 1) : a);
    b = b > BJ_K - 1 ? b - (BJ_K - 1) : b;
    lo = min(a, b);
    hi = max(a, b);
}
__device__ __forceinline__ void bj_inner_all(BjShared& S, float tol, float noise) {
    const int tid = threadIdx.x;
    for (int e = tid; e < BJ_K * BJ_K; e += BJ_SOLVERS) S.Q[0][(e >> 5) * BJ_QLD + (e & 31)] = (e >> 5) == (e & 31);
    const int bi = tid >> 4, bj = tid & 15, qa = 4 * (tid & 3);
    float* Qr = S.Q[0] + (tid >> 2) * BJ_QLD;
    int cur = 0;
    bj_sync_some<BJ_SOLVERS>();
    for (int rnd = 0; rnd < BJ_K - 1; ++rnd) {
        const float* G = S.G[cur];
        int p[2], q[2], p1, q1, qu[4], qv[4];
        bj_pair(rnd, bj, p1, q1);
        const float gpp = G[p1 * BJ_GLD + p1], gqq = G[q1 * BJ_GLD + q1], gpq = G[p1 * BJ_GLD + q1];
        float a[2], b[2], c[2], d[2], x[4], y[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            bj_pair(rnd, bi + 8 * h, p[h], q[h]);
            a[h] = G[p[h] * BJ_GLD + p1];
            b[h] = G[p[h] * BJ_GLD + q1];
            c[h] = G[q[h] * BJ_GLD + p1];
            d[h] = G[q[h] * BJ_GLD + q1];
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            bj_pair(rnd, qa + h, qu[h], qv[h]);
            x[h] = Qr[qu[h]];
            y[h] = Qr[qv[h]];
        }
        float cj, sj;
        if (!bj_decide(gpp, gqq, gpq, tol, noise, cj, sj)) continue;   // (the same in every warp)
        float* H = S.G[cur ^ 1];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float ci = __shfl_sync(0xffffffffu, cj, bi + 8 * h), si = __shfl_sync(0xffffffffu, sj, bi + 8 * h);
            // columns (p1, q1) by (cj, sj), then rows (p, q) by (ci, si)
            const float a1 = cj * a[h] - sj * b[h], b1 = sj * a[h] + cj * b[h];
            const float c1 = cj * c[h] - sj * d[h], d1 = sj * c[h] + cj * d[h];
            H[p[h] * BJ_GLD + p1] = ci * a1 - si * c1;
            H[q[h] * BJ_GLD + p1] = si * a1 + ci * c1;
            H[p[h] * BJ_GLD + q1] = ci * b1 - si * d1;
            H[q[h] * BJ_GLD + q1] = si * b1 + ci * d1;
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float cq = __shfl_sync(0xffffffffu, cj, qa + h), sq = __shfl_sync(0xffffffffu, sj, qa + h);
            Qr[qu[h]] = cq * x[h] - sq * y[h];
            Qr[qv[h]] = sq * x[h] + cq * y[h];
        }
        cur ^= 1;
        bj_sync_some<BJ_SOLVERS>();
    }
    if (tid == 0) S.cur = cur;
}

// One pass over the 256 pairs of a column of block I with one of block J, 16 rounds: pair i of round r is
// (i, 16 + (i + r) % 16).  G is symmetric and the first halves of the pairs never move, so a thread
// keeps its two elements of the I x I block in registers and only the I x J and J x J blocks (and the
// diagonal) go through shared memory.  Q belongs to a fifth warp, a row per lane in registers (the J
// half is kept rotated so that pair i's column is q[16 + i]).
__device__ __forceinline__ void bj_inner_cross(BjShared& S, float tol, float noise) {
    const int tid = threadIdx.x, bi = tid >> 4, bj = tid & 15;
    float ll[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) ll[h] = S.G[0][(bi + 8 * h) * BJ_GLD + bj];
    int cur = 0;
    for (int rnd = 0; rnd < BJ_B; ++rnd) {
        const float* G = S.G[cur];
        const int q1 = BJ_B + ((bj + rnd) & (BJ_B - 1));
        const float gpp = G[bj * BJ_GLD + bj], gqq = G[q1 * BJ_GLD + q1], gpq = G[bj * BJ_GLD + q1];
        float b[2], c[2], d[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int p = bi + 8 * h, q = BJ_B + ((p + rnd) & (BJ_B - 1));
            b[h] = G[p * BJ_GLD + q1];
            c[h] = G[bj * BJ_GLD + q];
            d[h] = G[q * BJ_GLD + q1];
        }
        float cj, sj;
        if (!bj_decide(gpp, gqq, gpq, tol, noise, cj, sj)) continue;   // (the same in every warp)
        float* H = S.G[cur ^ 1];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int p = bi + 8 * h, q = BJ_B + ((p + rnd) & (BJ_B - 1));
            const float ci = __shfl_sync(0xffffffffu, cj, p), si = __shfl_sync(0xffffffffu, sj, p);
            const float a1 = cj * ll[h] - sj * b[h], b1 = sj * ll[h] + cj * b[h];
            const float c1 = cj * c[h] - sj * d[h], d1 = sj * c[h] + cj * d[h];
            ll[h] = ci * a1 - si * c1;
            H[p * BJ_GLD + q1] = ci * b1 - si * d1;
            H[q * BJ_GLD + q1] = si * b1 + ci * d1;
            if (p == bj) H[p * BJ_GLD + p] = ll[h];
        }
        cur ^= 1;
        bj_sync_some<BJ_SOLVERS + 32>();
    }
    if (tid == 0) S.cur = cur;
}
__device__ __forceinline__ void bj_inner_cross_q(const BjShared& S, float tol, float noise, float (&q)[BJ_K]) {
    const int lane = threadIdx.x & 31, bj = lane & 15;
#pragma unroll
    for (int u = 0; u < BJ_K; ++u) q[u] = u == lane ? 1.f : 0.f;
    int cur = 0;
    for (int rnd = 0; rnd < BJ_B; ++rnd) {
        const float* G = S.G[cur];
        const int q1 = BJ_B + ((bj + rnd) & (BJ_B - 1));
        const float gpp = G[bj * BJ_GLD + bj], gqq = G[q1 * BJ_GLD + q1], gpq = G[bj * BJ_GLD + q1];
        float cj, sj;
        const bool any = bj_decide(gpp, gqq, gpq, tol, noise, cj, sj);
        if (any) {
            cur ^= 1;
            bj_sync_some<BJ_SOLVERS + 32>();         // before Q's rotations: the solvers need not wait for them
#pragma unroll
            for (int i = 0; i < BJ_B; ++i) {
                const float c = __shfl_sync(0xffffffffu, cj, i), sn = __shfl_sync(0xffffffffu, sj, i);
                const float x = q[i], y = q[BJ_B + i];
                q[i] = c * x - sn * y;
                q[BJ_B + i] = sn * x + c * y;
            }
        }
        const float first = q[BJ_B];
#pragma unroll
        for (int i = BJ_B; i < BJ_K - 1; ++i) q[i] = q[i + 1];
        q[BJ_K - 1] = first;
    }
}

// Block pair (I, J), I < J, of position pi in a round; false: one of the two is padding.  (One block: the
// pair (0, 0) of round 0.)
__device__ __forceinline__ bool bj_blocks(const BjSec& b, int pi, int round, int& I, int& J) {
    I = J = 0;
    if (b.nb == 1) return round == 0;
    if (round >= b.nbp - 1) return false;
    I = rr_pos(pi, round, b.nbp);
    J = rr_pos(b.nbp - 1 - pi, round, b.nbp);
    if (I > J) { const int t = I; I = J; J = t; }
    return J < b.nb;
}
// Pairs that block x has been in before (sweep, round): every round but, with an odd number of blocks,
// the one it sits out (round 0 for block 0, else the r with 2 r = x modulo nbp - 1).
__device__ __forceinline__ int bj_earlier(const BjSec& b, int x, int sweep, int round) {
    if (b.nb == 1) return sweep;
    if ((b.nb & 1) == 0) return sweep * (b.nbp - 1) + round;
    const int out = x == 0 ? 0 : ((x & 1) ? (x + b.nbp - 1) / 2 : x / 2);
    return sweep * (b.nbp - 2) + round - (out < round ? 1 : 0);
}

// The queue's ordering words.  wdone[block]: pairs of the block whose W columns are final; vdone[block]:
// stamp of the block's last finished rotation of V.
struct BjOrder {
    int* wdone;
    int* vdone;
    int* abort_flag;
    unsigned* err;
};
// Bounded wait (one thread) until *word >= value; false: gave up (the abort flag and ERRBIT_TIMEOUT are
// set) or another CTA has, or *stop became nonzero (then *stopped).
__device__ __forceinline__ bool bj_wait(const int* word, int value, const BjOrder& o, const int* stop, bool* stopped) {
    uint64_t t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    while (*((volatile const int*)word) < value) {
        if (*((volatile int*)o.abort_flag) != 0) return false;
        if (stop && *((volatile const int*)stop) != 0) {
            *stopped = true;
            return false;
        }
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > 2000000000ull) {
            atomicOr(o.err, ERRBIT_TIMEOUT);
            atomicExch(o.abort_flag, 1);
            return false;
        }
    }
    return true;
}

// The block pair (I, J).  Returns (in every thread) the FP32 flops of its Gram matrix and, if it rotated,
// of the column rotations (negative when it rotated: -flops), 0 when it is known to be converged.  X
// holds `cap` staged rows: a sector up to that is staged once, a taller one is streamed in row chunks
// (its W is read twice: once for the Gram matrix, once for the rotation).
// With `order` (the queue) the W columns are published before V's are rotated: the next pairs of these
// blocks need W only, so V is off the chain of rounds; V's rotations of a block follow each other by
// their stamps.
__device__ double bj_task(BjShared& S, float* __restrict__ X, int cap, const SvdSec& s, const BjSec& b, int si, int I,
                          int J, int round, float* __restrict__ W, float* __restrict__ V, float tol, float noise_c,
                          float* __restrict__ gmax, int* __restrict__ bmod, int* __restrict__ pchk, int now,
                          const BjOrder* order, int doneI, int doneJ) {
    const int cI = I * BJ_B, kI = min(BJ_B, s.n - cI), cJ = J * BJ_B, kJ = I == J ? 0 : min(BJ_B, s.n - cJ);
    // skip a pair found converged after both blocks' last rotations (same values in every thread)
    int* const chk = pchk + b.pst0 + I * b.nb + J;
    const int modI = __ldcg(bmod + b.blk0 + I), modJ = __ldcg(bmod + b.blk0 + J);
    if (__ldcg(chk) > max(modI, modJ)) return 0.0;
    const int k = kI + kJ;
    const int tid = threadIdx.x, lane = tid & 31;
    const double gram_flops = 2.0 * s.p * k * k, rot_flops = 2.0 * ((double)s.p + s.n) * k * k;
    const bool resident = s.p <= cap;                 // W's columns fit: staged once
    const int ldx = bj_ldx(min(s.p, cap));
    if (tid < BJ_K) S.gcol[tid] = tid < kI ? cI + tid : (tid < k ? cJ + tid - kI : -1);
    if (tid == 0) S.gmax = *((volatile float*)&gmax[si]);
    __syncthreads();
    float* const Ws = W + s.w_off;
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int r0 = 0; r0 < s.p; r0 += cap) {
        const int len = min(cap, s.p - r0);
        bj_stage(X, ldx, Ws, s.p, r0, len, S.gcol);
        cp_async_wait_all();
        __syncthreads();
        bj_gram_acc(acc, X, ldx, len);
        if (!resident) __syncthreads();
    }
    bj_gram_reduce(S, acc);
    const float* G = S.G[0];
    // the sector's rounding level, from the largest squared column norm it has seen
    float dmax = G[lane * BJ_GLD + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (tid == 0 && dmax > S.gmax) atomicMax(reinterpret_cast<int*>(&gmax[si]), __float_as_int(dmax));
    const float noise = noise_c * sqrtf(fmaxf(dmax, S.gmax));
    // pairs that need a rotation: inside a block (1), across (2)
    int need = 0;
    for (int e = tid; e < BJ_K * BJ_K; e += BJ_THREADS) {
        const int u = e >> 5, v = e & 31;
        if (u < v && v < k && bj_need(G[u * BJ_GLD + v], G[u * BJ_GLD + u], G[v * BJ_GLD + v], tol, noise))
            need |= u < BJ_B && v >= BJ_B ? 2 : 1;
    }
    const int across = __syncthreads_or(need & 2);
    // all pairs once a sweep for every block: in round 0, in round 1 for the block that sits out round
    // 0 (block 0 of an odd number)
    const bool whole = round == 0 || (round == 1 && (b.nb & 1) && I == 0);
    if (!across && !__syncthreads_or(need)) {
        if (tid == 0) *chk = now;
        return gram_flops;
    }
    const bool cross = across && !whole;
    float q[BJ_K];                                     // the fifth warp's rows of Q (cross)
    if (cross) {
        if (tid < BJ_SOLVERS) bj_inner_cross(S, tol, noise);
        else if (tid < BJ_SOLVERS + 32) bj_inner_cross_q(S, tol, noise, q);
    } else if (tid < BJ_SOLVERS) {
        bj_inner_all(S, tol, noise);
    }
    __syncthreads();
    // order the eigenvectors of the k real columns by decreasing eigenvalue (ties: lower index
    // first); the padding columns are never rotated and keep their positions k..31 (a real
    // column of a numerically rank-deficient pair can end with an eigenvalue rounded below zero,
    // which must not trade places with a padding column's zero)
    if (tid < BJ_K) {
        const float* Gf = S.G[S.cur];
        const float d = Gf[tid * BJ_GLD + tid];
        int r = tid;
        if (tid < k) {
            r = 0;
            for (int v = 0; v < k; ++v) {
                const float e = Gf[v * BJ_GLD + v];
                r += (e > d) || (e == d && v < tid);
            }
        }
        S.pos[tid] = r;
    }
    __syncthreads();
    float* Qp = S.Q[1];
    if (cross) {
        if (tid >= BJ_SOLVERS && tid < BJ_SOLVERS + 32)
#pragma unroll
            for (int u = 0; u < BJ_K; ++u) Qp[lane * BJ_QLD + S.pos[u]] = q[u];
    } else {
        for (int e = tid; e < BJ_K * BJ_K; e += BJ_THREADS) {
            const int u = e >> 5, v = e & 31;
            Qp[u * BJ_QLD + S.pos[v]] = S.Q[0][u * BJ_QLD + v];
        }
    }
    __syncthreads();
    for (int r0 = 0; r0 < s.p; r0 += cap) {
        const int len = min(cap, s.p - r0);
        if (!resident) {
            bj_stage(X, ldx, Ws, s.p, r0, len, S.gcol);
            cp_async_wait_all();
            __syncthreads();
        }
        bj_rotate_out(X, ldx, len, Qp, Ws, s.p, r0, S.gcol, k);
        __syncthreads();
    }
    if (tid == 0) {
        bmod[b.blk0 + I] = now;
        bmod[b.blk0 + J] = now;
        if (order) {
            __threadfence();                           // every thread's columns (barrier) and the stamps
            *((volatile int*)order->wdone + b.blk0 + I) = doneI + 1;
            *((volatile int*)order->wdone + b.blk0 + J) = doneJ + 1;
            // (the abort flag ends the wait: the results are void then)
            if (bj_wait(order->vdone + b.blk0 + I, modI, *order, nullptr, nullptr))
                bj_wait(order->vdone + b.blk0 + J, modJ, *order, nullptr, nullptr);
            __threadfence();
        }
    }
    __syncthreads();
    // V's columns take the same way
    for (int r0 = 0; r0 < s.n; r0 += cap) {
        const int len = min(cap, s.n - r0);
        bj_stage(X, ldx, V + s.v_off, s.n, r0, len, S.gcol);
        cp_async_wait_all();
        __syncthreads();
        bj_rotate_out(X, ldx, len, Qp, V + s.v_off, s.n, r0, S.gcol, k);
        __syncthreads();
    }
    if (order && tid == 0) {
        __threadfence();
        *((volatile int*)order->vdone + b.blk0 + I) = now;
        *((volatile int*)order->vdone + b.blk0 + J) = now;
    }
    return -(gram_flops + rot_flops);
}

// One round of one sweep: every CTA takes tasks blockIdx.x, blockIdx.x + gridDim.x, ...
// rot[sweep] counts the pairs rotated in this sweep (zeroed by the host).  A launch whose previous
// sweep rotated nothing returns at once (the host enqueues a sweep before it has read the result
// of the one before).
__global__ void __launch_bounds__(BJ_THREADS, 2)
    k_bjacobi_round(const SvdSec* __restrict__ secs, const BjSec* __restrict__ bsecs, const int* __restrict__ task_sec,
                    int ntasks, int round, int sweep, int nrounds, int cap, float* __restrict__ W,
                    float* __restrict__ V, float noise_c, float* __restrict__ gmax, int* __restrict__ bmod,
                    int* __restrict__ pchk, int* __restrict__ rot, unsigned long long* __restrict__ flops) {
    extern __shared__ __align__(16) unsigned char bj_smem[];
    if (sweep > 0 && *((volatile int*)&rot[sweep - 1]) == 0) return;
    BjShared& S = *reinterpret_cast<BjShared*>(bj_smem);
    float* X = reinterpret_cast<float*>(bj_smem + sizeof(BjShared));
    double fl = 0.0;
    for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
        const int si = task_sec[t];
        const SvdSec s = secs[si];
        const BjSec b = bsecs[si];
        int I, J;
        if (!bj_blocks(b, t - b.task0, round, I, J)) continue;
        const double r = bj_task(S, X, cap, s, b, si, I, J, round, W, V, b.tol, noise_c, gmax, bmod, pchk,
                                 sweep * nrounds + round + 1, nullptr, 0, 0);
        fl += fabs(r);
        if (r < 0.0 && threadIdx.x == 0) atomicAdd(&rot[sweep], 1);
        __syncthreads();
    }
    if (threadIdx.x == 0 && fl > 0.0) atomicAdd(flops, (unsigned long long)fl);
}

// All sweeps in one cooperative launch, for a caller that has the GPU to itself, without grid-wide
// barriers.  Work items (sweep, round, sector, pair) are taken in order from one counter: per sweep
// the rounds in order, in each round every sector's pairs (taller sectors first).  An item waits only
// for the earlier pairs of its own two blocks (their W columns): blocks run ahead of each other within
// a sector, small sectors into later sweeps while the tall sectors' long round sequences are in
// flight.  Items depend on earlier items only and every CTA is resident, so the queue always drains: a
// CTA draws its next item while it works on one (the draw's latency is hidden), and the smallest
// unfinished item is always one being worked on, since its holder works on no smaller one.  V's
// rotations wait for rotations of earlier items likewise.  A sector whose sweep rotated nothing has
// converged: its later items are counted without work, and the launch ends once every sector has
// converged (or after max_sweeps; nact = sectors with columns).  Every wait is bounded
// (ERRBIT_TIMEOUT and the abort flag after 2 s).
// qstate (zeroed): [0] next item, [1] converged sectors, [2] abort flag, then converged flags (nsec),
// pairs rotated and items finished per sector and sweep (nsec x max_sweeps each).
// border (zeroed): wdone and vdone of every block (see BjOrder).  rot[sweep]: pairs rotated in that
// sweep over all sectors; *sweeps: sweeps run by the slowest sector.
__global__ void __launch_bounds__(BJ_THREADS, 2)
    k_bjacobi_queue(const SvdSec* __restrict__ secs, const BjSec* __restrict__ bsecs, const int2* __restrict__ items,
                    int per_sweep, int nsec, int nact, int nrounds, int max_sweeps, int cap,
                    float* __restrict__ W, float* __restrict__ V, float noise_c, float* __restrict__ gmax,
                    int* __restrict__ bmod, int* __restrict__ pchk, int* __restrict__ border, int nblk,
                    int* __restrict__ qstate, int* __restrict__ rot, int* __restrict__ sweeps,
                    unsigned* __restrict__ err, unsigned long long* __restrict__ flops) {
    extern __shared__ __align__(16) unsigned char bj_smem[];
    BjShared& S = *reinterpret_cast<BjShared*>(bj_smem);
    float* X = reinterpret_cast<float*>(bj_smem + sizeof(BjShared));
    const int tid = threadIdx.x;
    int* const qnext = qstate;
    int* const nconv = qstate + 1;
    int* const abort_flag = qstate + 2;
    int* const conv = qstate + 3;
    int* const srot = conv + nsec;
    int* const sdone = srot + nsec * max_sweeps;
    const BjOrder order = {border, border + nblk, abort_flag, err};
    const int total = per_sweep * max_sweeps;        // below 2^31 (checked by the host)
    double fl = 0.0;
    int next = 0;
    if (tid == 0) next = atomicAdd(qnext, 1);
    for (;;) {
        if (tid == 0) {
            S.qitem = next;
            if (next < total) {
                const int sweep = next / per_sweep;
                const int2 it = items[next - sweep * per_sweep];
                S.qsec = it.x;
                S.qsweep = sweep;
                S.qround = it.y >> 16;
                S.qpair = it.y & 0xffff;
            }
        }
        __syncthreads();
        if (S.qitem >= total) break;                 // uniform: read before anyone writes it again
        const int si = S.qsec, sweep = S.qsweep, round = S.qround, pi = S.qpair;
        const BjSec b = bsecs[si];
        const int nr = b.nb == 1 ? 1 : b.nbp - 1;
        int I, J;
        const bool real = bj_blocks(b, pi, round, I, J);
        const int doneI = bj_earlier(b, I, sweep, round), doneJ = bj_earlier(b, J, sweep, round);
        if (tid == 0) {
            next = atomicAdd(qnext, 1);              // used in the next turn of the loop
            int state = real ? 1 : 0;                // 1: work, 0: count only, -1: count and leave
            if (*((volatile int*)abort_flag) != 0 || *((volatile int*)nconv) >= nact) state = -1;
            else if (*((volatile int*)&conv[si]) != 0) state = 0;
            if (state == 1) {
                // both blocks' earlier pairs; or the sector has converged meanwhile (items of it that
                // leaving CTAs had drawn are not counted)
                bool stopped = false;
                if (!bj_wait(order.wdone + b.blk0 + I, doneI, order, &conv[si], &stopped) ||
                    !bj_wait(order.wdone + b.blk0 + J, doneJ, order, &conv[si], &stopped))
                    state = stopped ? 0 : -1;
                // the blocks' earlier pairs (columns, stamps) happen before this item's loads
                __threadfence();
            }
            S.qok = state;
        }
        __syncthreads();
        const int state = S.qok;
        bool rotated = false;
        if (state == 1) {
            const SvdSec s = secs[si];
            const double r = bj_task(S, X, cap, s, b, si, I, J, round, W, V, b.tol, noise_c, gmax, bmod, pchk,
                                     sweep * nrounds + round + 1, &order, doneI, doneJ);
            fl += fabs(r);
            if (tid == 0) {
                rotated = r < 0.0;
                if (rotated) {
                    atomicAdd(&srot[si * max_sweeps + sweep], 1);
                    atomicAdd(&rot[sweep], 1);
                }
            }
        }
        __syncthreads();                             // every thread's reads and writes precede the counts
        if (tid == 0) {
            __threadfence();
            if (state == 1 && !rotated) {            // (a rotating pair published its columns itself)
                *((volatile int*)order.wdone + b.blk0 + I) = doneI + 1;
                *((volatile int*)order.wdone + b.blk0 + J) = doneJ + 1;
            }
            const int old = atomicAdd(&sdone[si * max_sweeps + sweep], 1);
            if (old + 1 == nr * b.ntask) {           // the last item of this sector's sweep
                __threadfence();
                if (*((volatile int*)&conv[si]) == 0) {
                    atomicMax(sweeps, sweep + 1);
                    // (two sweeps' last items may come here at once: the sector counts once)
                    if (*((volatile int*)&srot[si * max_sweeps + sweep]) == 0 && atomicExch(&conv[si], 1) == 0)
                        atomicAdd(nconv, 1);
                }
            }
        }
        if (state < 0) break;
    }
    if (tid == 0 && fl > 0.0) atomicAdd(flops, (unsigned long long)fl);
}

}  // namespace

void launch_bjacobi(const SvdSec* secs, const BjSec* bsecs, const int* task_sec, int ntasks, int nrounds, int max_rows,
                    int max_sweeps, float* W, float* V, float noise_c, float* gmax, int* bmod, int* pchk, int* border,
                    int nblk, int* rot, int* sweeps, unsigned* err, unsigned long long* flops, const int2* items,
                    int per_sweep, int nsec, int nact, int* qstate, cudaStream_t st) {
    if (ntasks <= 0 || nrounds <= 0) {
        PD_CK(cudaMemsetAsync(sweeps, 0, sizeof(int), st));
        return;
    }
    // Two CTAs share an SM while the tallest sector's columns fit in half of it: each hides the other's
    // barriers and latencies (mixed-mode cylinder bond m = 2000: 40.1 ms a split, 45.9 with one an SM; with
    // fewer tasks than SMs no difference).  Taller ones get the SM, or are streamed through it in row
    // chunks, which reads a column twice.
    const int cap = std::max(32, max_rows <= bj_fit(2) ? std::min(max_rows, bj_fit(2)) : std::min(max_rows, bj_fit(1)));
    const size_t smem = sizeof(BjShared) + (size_t)bj_ldx(cap) * BJ_K * sizeof(float);
    constexpr int BJ_SMEM_MAX = (int)sizeof(BjShared) + bj_ldx(bj_fit(1)) * BJ_K * (int)sizeof(float);
    // the shared-memory ceiling is raised once per process to the largest size any launch uses
    // (region threads launch concurrently with different sizes)
    static const cudaError_t attr =
        cudaFuncSetAttribute(k_bjacobi_round, cudaFuncAttributeMaxDynamicSharedMemorySize, BJ_SMEM_MAX);
    PD_CK(attr);
    int dev = 0, sms = 0;
    PD_CK(cudaGetDevice(&dev));
    PD_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (g_sm_cap == 0) {
        // the GPU is this caller's: all sweeps in one cooperative launch (the dependency queue)
        static const cudaError_t attr_c =
            cudaFuncSetAttribute(k_bjacobi_queue, cudaFuncAttributeMaxDynamicSharedMemorySize, BJ_SMEM_MAX);
        PD_CK(attr_c);
        int per_sm = 0;
        PD_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bjacobi_queue, BJ_THREADS, smem));
        PD_REQUIRE(per_sm > 0, DMRG_ERR_CAPACITY, "block Jacobi: kernel does not fit on an SM");
        const int cblocks = std::max(1, std::min(per_sweep, per_sm * sms));
        PD_CK(cudaMemsetAsync(sweeps, 0, sizeof(int), st));
        void* args[] = {(void*)&secs, (void*)&bsecs, (void*)&items, (void*)&per_sweep, (void*)&nsec, (void*)&nact,
                        (void*)&nrounds, (void*)&max_sweeps, (void*)&cap, (void*)&W, (void*)&V, (void*)&noise_c,
                        (void*)&gmax, (void*)&bmod, (void*)&pchk, (void*)&border, (void*)&nblk, (void*)&qstate,
                        (void*)&rot, (void*)&sweeps, (void*)&err, (void*)&flops};
        PD_CK(cudaLaunchCooperativeKernel((void*)k_bjacobi_queue, cblocks, BJ_THREADS, args, smem, st));
        PD_LAUNCHED();
        return;
    }
    // regions run concurrently: one launch per round, nothing spins
    const int blocks = std::max(1, std::min(ntasks, 4 * sms));
    // rounds are enqueued sweep by sweep; the host reads rot of sweep s - 1 after enqueuing sweep s
    // (pinned copy + event), so the device never waits for the host; a sweep enqueued after the
    // converged one returns at once.
    int* hrot = sweep_flags_host(max_sweeps);
    std::vector<cudaEvent_t> evs(max_sweeps, nullptr);
    int done = max_sweeps;
    try {
        for (int sweep = 0; sweep < max_sweeps; ++sweep) {
            for (int round = 0; round < nrounds; ++round) {
                k_bjacobi_round<<<blocks, BJ_THREADS, smem, st>>>(secs, bsecs, task_sec, ntasks, round, sweep,
                                                                   nrounds, cap, W, V,
                                                                   noise_c, gmax, bmod, pchk, rot, flops);
                PD_LAUNCHED();
            }
            PD_CK(cudaMemcpyAsync(hrot + sweep, rot + sweep, sizeof(int), cudaMemcpyDeviceToHost, st));
            PD_CK(cudaEventCreateWithFlags(&evs[sweep], cudaEventDisableTiming));
            PD_CK(cudaEventRecord(evs[sweep], st));
            if (sweep > 0) {
                PD_CK(cudaEventSynchronize(evs[sweep - 1]));
                if (hrot[sweep - 1] == 0) {
                    done = sweep;      // sweep - 1 rotated nothing; the launches of `sweep` exit at once
                    break;
                }
            }
        }
        if (done == max_sweeps) {
            PD_CK(cudaEventSynchronize(evs[max_sweeps - 1]));
            if (hrot[max_sweeps - 1] == 0) done = max_sweeps;
        }
    } catch (...) {
        for (auto e : evs)
            if (e) cudaEventDestroy(e);
        throw;
    }
    for (auto e : evs)
        if (e) cudaEventDestroy(e);
    PD_CK(cudaMemcpyAsync(sweeps, &done, sizeof(int), cudaMemcpyHostToDevice, st));
}

}  // namespace pd
