// FP64 / memory-bound kernels of the two-site DMRG step.
//
//  * k_gemm_f64     grouped, strided FP64 GEMM (the parity-mode contractions of the projected
//                   Hamiltonian and of the projected-operator updates, Sec. II)
//  * k_copy/k_mix   block gathers, transposes, MPO channel mixing (memory-bound)
//  * k_diag         diagonal of the projected Hamiltonian (Davidson preconditioner)
//  * Davidson       dot products, Ritz vectors, residuals, Gram-Schmidt, small Jacobi eigensolver
//  * SVD            batched one-sided (Hestenes) Jacobi SVD per charge sector, Eq. (svd)
//  * truncation     global keep-largest-m selection over all sectors (single CTA)
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <type_traits>
#include <vector>

#include "grid_sync.cuh"
#include "internal.h"


namespace pd {

namespace {

template <class T>
__device__ __forceinline__ double to_d(T x) { return (double)x; }
template <>
__device__ __forceinline__ double to_d<__nv_bfloat16>(__nv_bfloat16 x) { return (double)__bfloat162float(x); }

template <class T>
__device__ __forceinline__ T from_d(double x) { return (T)x; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_d<__nv_bfloat16>(double x) { return __float2bfloat16_rn((float)x); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sum (blockDim.x multiple of 32, <= 1024); result valid in every thread.
__device__ double block_sum(double v) {
    __shared__ double red[32];
    __shared__ double total;
    v = warp_sum(v);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int nw = blockDim.x >> 5;
        double x = lane < nw ? red[lane] : 0.0;
        x = warp_sum(x);
        if (lane == 0) total = x;
    }
    __syncthreads();
    return total;
}

// ------------------------------------------------------------------------------------------
// Grouped FP64 GEMM.  This part issues 2 DFMA per clock and SM (one warp instruction every 64
// clocks per scheduler), so the FP64 pipe is the bound and everything else is sized around it:
//  * A warp owns a 16 x 16 output tile (a lane 2 rows x 4 columns) and skips the row octets and
//    column quads outside the block, so small charge blocks pay for at most 8 x 4 padding.
//    (64 x 64 CTA tiles computed their padding: a 15 x 15 block cost as much as a 64 x 64 one.)
//  * Operands come straight from L1 / L2 into registers, four k at a time and one group ahead:
//    a group is 32 DFMA = 2048 clocks of one scheduler, far above an L2 latency, and a 16-row
//    K-contiguous panel re-reads its 128-byte lines from L1.  No shared memory, no barriers.
//  * KS warps of a CTA share one tile with K (or the segments) split between them, summed in
//    warp order at the end, so that a few tiles still reach every scheduler (see f64_shape).
// FP64 matvec at the 24x8 cylinder's m = 500 bond, whole call: 3926 -> 1960 us; batches at f64_shape.
// ------------------------------------------------------------------------------------------
template <int MI, int NJ>
__device__ __forceinline__ void f64_span(const double* pa0, const double* pa1, long long sak, const double* pb,
                                         const int (&ob)[4], long long sbk, int n, double (&acc)[2][4]) {
    constexpr int U = 4;
    double a[U][MI], b[U][NJ];
    int k = 0;
    if (n >= U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u][0] = pa0[u * sak];
            if (MI > 1) a[u][MI - 1] = pa1[u * sak];
#pragma unroll
            for (int j = 0; j < NJ; ++j) b[u][j] = pb[u * sbk + ob[j]];
        }
    }
    for (; k + U <= n; k += U) {
        double a2[U][MI], b2[U][NJ];
        pa0 += U * sak;
        pa1 += U * sak;
        pb += U * sbk;
        const bool more = k + 2 * U <= n;
        if (more) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                a2[u][0] = pa0[u * sak];
                if (MI > 1) a2[u][MI - 1] = pa1[u * sak];
#pragma unroll
                for (int j = 0; j < NJ; ++j) b2[u][j] = pb[u * sbk + ob[j]];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = fma(a[u][i], b[u][j], acc[i][j]);
        if (more) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int i = 0; i < MI; ++i) a[u][i] = a2[u][i];
#pragma unroll
                for (int j = 0; j < NJ; ++j) b[u][j] = b2[u][j];
            }
        }
    }
    // the last n % U steps: loads first, then the products
    const int rem = n - k;
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
        if (u < rem) {
            a[u][0] = pa0[u * sak];
            if (MI > 1) a[u][MI - 1] = pa1[u * sak];
#pragma unroll
            for (int j = 0; j < NJ; ++j) b[u][j] = pb[u * sbk + ob[j]];
        }
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
        if (u < rem)
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = fma(a[u][i], b[u][j], acc[i][j]);
}

// One warp's part of a tile: all segments (KS = 1), or the segments ks, ks + KS, ... when there are
// at least 4 KS of them, else the ks-th part of every segment's K.
template <int MI, int NJ, int KS>
__device__ __forceinline__ void f64_tile(const GProb& p, const GSeg* __restrict__ segs, const double* __restrict__ A,
                                         const double* __restrict__ B, int m0, int n0, int ks, double (&acc)[2][4]) {
    const int lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
    // rows and columns beyond the block read its last one; their results are not stored
    const long long ra0 = (long long)min(m0 + r, p.M - 1) * p.sam, ra1 = (long long)min(m0 + 8 + r, p.M - 1) * p.sam;
    const int nb = min(n0 + c, p.N - 1);
    int ob[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) ob[j] = (min(n0 + c + 4 * j, p.N - 1) - nb) * p.sbn;
    const bool whole = KS == 1 || p.nseg >= 4 * KS;
    for (int s = (KS > 1 && whole) ? ks : 0; s < p.nseg; s += (KS > 1 && whole) ? KS : 1) {
        const GSeg sg = segs[p.seg0 + s];
        int k0 = 0, k1 = sg.K;
        if (!whole) {
            k0 = (int)((long long)sg.K * ks / KS);
            k1 = (int)((long long)sg.K * (ks + 1) / KS);
        }
        const double* a = A + sg.a_off + (long long)k0 * p.sak;
        const double* b = B + sg.b_off + (long long)k0 * p.sbk + (long long)nb * p.sbn;
        f64_span<MI, NJ>(a + ra0, a + ra1, p.sak, b, ob, p.sbk, k1 - k0, acc);
    }
}

// tiles[blockIdx.x / sub]: a tile of `sub` CTA tiles (row by row, edge / CT of them side by side).
// KS = 1: CT = 32, four warps with a 16 x 16 tile each; KS > 1: CT = 16, KS warps on one tile.
template <int KS>
__global__ void __launch_bounds__(KS == 1 ? 128 : 32 * KS)
    k_gemm_f64(const GProb* __restrict__ probs, const GSeg* __restrict__ segs, const GTile* __restrict__ tiles, int side,
               const double* __restrict__ A, const double* __restrict__ B, double* __restrict__ C) {
    constexpr int CT = KS == 1 ? 32 : 16;
    __shared__ double part[KS > 1 ? KS - 1 : 1][KS > 1 ? 256 : 1];
    const int sub = side * side, si = blockIdx.x % sub;
    const GTile t = tiles[blockIdx.x / sub];
    const GProb p = probs[t.prob];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int m0 = t.m0 + (si / side) * CT, n0 = t.n0 + (si % side) * CT;
    if (KS == 1) {
        m0 += (warp >> 1) * 16;
        n0 += (warp & 1) * 16;
    }
    if (m0 >= p.M || n0 >= p.N) return;              // whole warps (KS = 1), whole CTAs (KS > 1)
    double acc[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
    const int ks = KS > 1 ? warp : 0;
    const int nj = min(4, (p.N - n0 + 3) / 4);
    if (p.M - m0 > 8) {
        if (nj == 4) f64_tile<2, 4, KS>(p, segs, A, B, m0, n0, ks, acc);
        else if (nj == 3) f64_tile<2, 3, KS>(p, segs, A, B, m0, n0, ks, acc);
        else if (nj == 2) f64_tile<2, 2, KS>(p, segs, A, B, m0, n0, ks, acc);
        else f64_tile<2, 1, KS>(p, segs, A, B, m0, n0, ks, acc);
    } else {
        if (nj == 4) f64_tile<1, 4, KS>(p, segs, A, B, m0, n0, ks, acc);
        else if (nj == 3) f64_tile<1, 3, KS>(p, segs, A, B, m0, n0, ks, acc);
        else if (nj == 2) f64_tile<1, 2, KS>(p, segs, A, B, m0, n0, ks, acc);
        else f64_tile<1, 1, KS>(p, segs, A, B, m0, n0, ks, acc);
    }
    if (KS > 1) {
        if (warp > 0)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) part[warp - 1][(i * 4 + j) * 32 + lane] = acc[i][j];
        __syncthreads();
        if (warp > 0) return;
#pragma unroll
        for (int w = 0; w < KS - 1; ++w)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] += part[w][(i * 4 + j) * 32 + lane];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int m = m0 + (lane >> 2) + 8 * i;
        if (m >= p.M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + (lane & 3) + 4 * j;
            if (n >= p.N) continue;
            const long long idx = p.c_off + (long long)m * p.scm + (long long)n * p.scn;
            double v = p.alpha * acc[i][j];
            if (p.accumulate) v += C[idx];
            C[idx] = v;
        }
    }
}

// ------------------------------------------------------------------------------------------
// Grouped FP32 GEMM (mixed-mode environments, refinement matvec) on the FMA units, which bound it:
// 64 x 64 output tile per CTA of two warps, 8 x 8 values per thread, so a step in k is 64 FMA on four
// 16-byte shared loads.  64 x 64 loses least to the blocks' edges (sectors of 40-320 states), and a
// warp whose 32 rows lie outside the block does no products.  Operands are K-major slabs whose rows
// are zero up to a multiple of 16 in k (the tensor-core layout): they come in as float4 along k, one
// chunk of 16 ahead in registers, and are stored k-major into a double buffer -- one barrier a chunk.
// Each value is one chain of FMA in k order, as in the 4 x 4 kernel before: the same bits.
// FP32 environment update at the 24x8 cylinder's m = 2000 bond, its two GEMMs (23 GFLOP): 1125 us with 4 x 4
// values a thread, 603 now (38 TFLOP/s of the 78.5 measured; the rest is blocks' edges).
// ------------------------------------------------------------------------------------------
constexpr int F32_T = 64, F32_K = 16, F32_LD = F32_T + 4;
__global__ void __launch_bounds__(64) k_gemm_f32(const GProb* __restrict__ probs, const GSeg* __restrict__ segs,
                                                 const GTile* __restrict__ tiles, const float* __restrict__ A,
                                                 const float* __restrict__ B, float* __restrict__ C) {
    __shared__ __align__(16) float As[2][F32_K][F32_LD], Bs[2][F32_K][F32_LD];
    const GTile t = tiles[blockIdx.x];
    const GProb p = probs[t.prob];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tr = 32 * warp + 4 * (lane >> 3), tc = 4 * (lane & 7);   // rows tr..+3, tr+16..; cols tc..+3, tc+32..
    // loader: four threads take the 64 bytes of a row's chunk, 16 rows a pass (rows outside the block are
    // clamped into it and not stored).  A row's values go to columns row ^ 8 in the upper half of the
    // chunk, which keeps these transposing stores free of bank conflicts.
    const int lr = tid >> 2, lk = 4 * (tid & 3), sw = lr ^ (lk & 8);
    long long ra[4], rb[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ra[q] = (long long)min(t.m0 + lr + 16 * q, p.M - 1) * p.sam + lk;
        rb[q] = (long long)min(t.n0 + lr + 16 * q, p.N - 1) * p.sbn + lk;
    }
    const bool busy = t.m0 + 32 * warp < p.M;
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    float4 fa[4], fb[4];
    int sgi = 0, k0 = 0, buf = 0;
    GSeg sg = segs[p.seg0];
    auto load = [&]() {
        const float* a = A + sg.a_off + k0;
        const float* b = B + sg.b_off + k0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            fa[q] = *reinterpret_cast<const float4*>(a + ra[q]);
            fb[q] = *reinterpret_cast<const float4*>(b + rb[q]);
        }
    };
    auto store = [&](int to) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            As[to][lk][sw + 16 * q] = fa[q].x;
            As[to][lk + 1][sw + 16 * q] = fa[q].y;
            As[to][lk + 2][sw + 16 * q] = fa[q].z;
            As[to][lk + 3][sw + 16 * q] = fa[q].w;
            Bs[to][lk][sw + 16 * q] = fb[q].x;
            Bs[to][lk + 1][sw + 16 * q] = fb[q].y;
            Bs[to][lk + 2][sw + 16 * q] = fb[q].z;
            Bs[to][lk + 3][sw + 16 * q] = fb[q].w;
        }
    };
    load();
    store(0);
    __syncthreads();
    for (;;) {
        // next chunk: this segment's next 16, or the next segment's first
        k0 += F32_K;
        if (k0 >= sg.K) {
            k0 = 0;
            if (++sgi < p.nseg) sg = segs[p.seg0 + sgi];
        }
        const bool more = sgi < p.nseg;
        if (more) load();
        if (busy) {
#pragma unroll
            for (int k = 0; k < F32_K; ++k) {
                const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][k][tr ^ (k & 8)]);
                const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][k][(tr + 16) ^ (k & 8)]);
                const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][k][tc ^ (k & 8)]);
                const float4 b1 = *reinterpret_cast<const float4*>(&Bs[buf][k][(tc + 32) ^ (k & 8)]);
                const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
            }
        }
        if (!more) break;
        buf ^= 1;
        store(buf);
        __syncthreads();
    }
    if (!busy) return;
    const float alpha = (float)p.alpha;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int n = t.n0 + tc + (j & 3) + (j >> 2) * 32;
        if (n >= p.N) continue;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int m = t.m0 + tr + (i & 3) + (i >> 2) * 16;
            if (m >= p.M) continue;
            const long long idx = p.c_off + (long long)m * p.scm + (long long)n * p.scn;
            float v = alpha * acc[i][j];
            if (p.accumulate) v += C[idx];
            C[idx] = v;
        }
    }
}

// ------------------------------------------------------------------------------------------
// Block copies, MPO channel mixing, diagonal
// ------------------------------------------------------------------------------------------
// Arithmetic of an element-wise kernel: FP64 when it writes FP64, else FP32 (an FP32 or bf16 output
// cannot hold more; the FP64 pipe of this part is 1/64 of the FP32 one and would otherwise bound
// these memory-bound kernels).
template <class Tin, class Tout>
using ew_t = typename std::conditional<std::is_same<Tout, double>::value, double, float>::type;
template <class A, class T>
__device__ __forceinline__ A to_a(T x) { return (A)x; }
template <>
__device__ __forceinline__ float to_a<float, __nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }
template <>
__device__ __forceinline__ double to_a<double, __nv_bfloat16>(__nv_bfloat16 x) { return (double)__bfloat162float(x); }
template <class T, class A>
__device__ __forceinline__ T from_a(A v) { return (T)v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_a<__nv_bfloat16, float>(float v) { return __float2bfloat16_rn(v); }
template <>
__device__ __forceinline__ __nv_bfloat16 from_a<__nv_bfloat16, double>(double v) { return __float2bfloat16_rn((float)v); }

// Row and column of element first + tid, + blockDim.x, ... of a rows x w job: two divisions a thread
// instead of one an element (element indices stay below 2^31 within a job).
struct ElemWalk {
    int r, c, dr, dc, w;
    __device__ __forceinline__ ElemWalk(int first, int width) : w(width) {
        const int e = first + (int)threadIdx.x;
        r = e / w;
        c = e - r * w;
        dr = (int)blockDim.x / w;
        dc = (int)blockDim.x - dr * w;
    }
    __device__ __forceinline__ void next() {
        r += dr;
        c += dc;
        if (c >= w) {
            c -= w;
            ++r;
        }
    }
};
// Elements a thread has in flight in the block kernels.  They are bound by memory latency (a chunk is a
// chain of list, job and data reads), so each thread issues its loads together; a chunk of 4096
// elements is two such groups.  Packing for one bf16 H_eff application of the 24x8 cylinder's m = 2000 bond
// (210 MB in all), with one load at a time and a division an element before: 162 -> 69 us; the mix of an
// environment update 81 -> 59.
constexpr int EW = 8;

template <class Tin, class Tout>
__global__ void __launch_bounds__(256) k_copy(const CopyJob* __restrict__ jobs, const int2* __restrict__ chunks,
                                              const Tin* __restrict__ src, Tout* __restrict__ dst) {
    using A = ew_t<Tin, Tout>;
    const int2 ch = chunks[blockIdx.x];
    const CopyJob j = jobs[ch.x];
    const int w = j.cols > j.zero_to ? j.cols : j.zero_to;
    const int len = (int)min((long long)j.rows * w - ch.y, (long long)CHUNK);
    const A scale = (A)j.scale;
    ElemWalk at(ch.y, w);
    for (int e = threadIdx.x; e < len; e += EW * blockDim.x) {
        A v[EW];
        long long d[EW];
#pragma unroll
        for (int u = 0; u < EW; ++u) {
            v[u] = A(0);
            d[u] = j.dst + (long long)at.r * j.drs + (long long)at.c * j.dcs;
            if (e + u * (int)blockDim.x < len && at.c < j.cols)
                v[u] = to_a<A>(src[j.src + (long long)at.r * j.srs + (long long)at.c * j.scs]);
            at.next();
        }
#pragma unroll
        for (int u = 0; u < EW; ++u)
            if (e + u * (int)blockDim.x < len) dst[d[u]] = from_a<Tout>(scale * v[u]);
    }
}

template <class Tin, class Tout>
__global__ void __launch_bounds__(256) k_mix(const MixJob* __restrict__ jobs, const int2* __restrict__ chunks,
                                             const MixTerm* __restrict__ terms, const Tin* __restrict__ in,
                                             Tout* __restrict__ out) {
    using A = ew_t<Tin, Tout>;
    const int2 ch = chunks[blockIdx.x];
    const MixJob j = jobs[ch.x];
    const int w = j.cols > j.zero_to ? j.cols : j.zero_to;
    const int len = (int)min((long long)j.rows * w - ch.y, (long long)CHUNK);
    ElemWalk at(ch.y, w);
    for (int e = threadIdx.x; e < len; e += EW * blockDim.x) {
        A v[EW];
        int r[EW], c[EW];
#pragma unroll
        for (int u = 0; u < EW; ++u) {
            v[u] = A(0);
            r[u] = at.r;
            c[u] = e + u * (int)blockDim.x < len ? at.c : -1;
            at.next();
        }
        for (int t = 0; t < j.nt; ++t) {
            const MixTerm tm = terms[j.t0 + t];
            const A coef = (A)tm.coef;
            A x[EW];
#pragma unroll
            for (int u = 0; u < EW; ++u)
                x[u] = (unsigned)c[u] < (unsigned)j.cols ? to_a<A>(in[tm.src + (long long)r[u] * tm.ld + c[u]]) : A(0);
#pragma unroll
            for (int u = 0; u < EW; ++u) v[u] += coef * x[u];
        }
#pragma unroll
        for (int u = 0; u < EW; ++u)
            if (c[u] >= 0) out[j.dst + (long long)r[u] * j.ldo + c[u]] = from_a<Tout>(c[u] < j.cols ? v[u] : A(0));
    }
}

template <class T>
__global__ void __launch_bounds__(256) k_diag(const DiagJob* __restrict__ jobs, const int2* __restrict__ chunks,
                                              const DiagTerm* __restrict__ terms, const T* __restrict__ Ls, int ldl,
                                              const T* __restrict__ Rs, int ldr, double* __restrict__ out) {
    const int2 ch = chunks[blockIdx.x];
    const DiagJob j = jobs[ch.x];
    const int len = (int)min((long long)j.rows * j.cols - ch.y, (long long)CHUNK);
    ElemWalk at(ch.y, j.cols);
    for (int e = threadIdx.x; e < len; e += EW * blockDim.x) {
        double v[EW];
        int r[EW], c[EW];
#pragma unroll
        for (int u = 0; u < EW; ++u) {
            v[u] = 0.0;
            const bool in = e + u * (int)blockDim.x < len;
            r[u] = in ? at.r : 0;
            c[u] = in ? at.c : 0;
            at.next();
        }
        for (int t = 0; t < j.nt; ++t) {
            const DiagTerm tm = terms[j.t0 + t];
#pragma unroll
            for (int u = 0; u < EW; ++u)
                v[u] += tm.coef * to_d(Ls[tm.l + (long long)r[u] * (ldl + 1)]) * to_d(Rs[tm.r + (long long)c[u] * (ldr + 1)]);
        }
#pragma unroll
        for (int u = 0; u < EW; ++u)
            if (e + u * (int)blockDim.x < len) out[j.off + ch.y + e + u * (int)blockDim.x] = v[u];
    }
}

// dst[i] = src[i], converted, i < n.
template <class Tin, class Tout>
__global__ void __launch_bounds__(256) k_convert(const Tin* __restrict__ src, Tout* __restrict__ dst, long long n) {
    using A = ew_t<Tin, Tout>;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += EW * step) {
        A v[EW];
#pragma unroll
        for (int u = 0; u < EW; ++u)
            if (e + u * step < n) v[u] = to_a<A>(src[e + u * step]);
#pragma unroll
        for (int u = 0; u < EW; ++u)
            if (e + u * step < n) dst[e + u * step] = from_a<Tout>(v[u]);
    }
}

// ------------------------------------------------------------------------------------------
// Dot product (FP64, deterministic two-pass reduction)
// ------------------------------------------------------------------------------------------
__global__ void k_dots_partial(const double* __restrict__ V, long long ldv, const double* __restrict__ y,
                               long long n, double* __restrict__ partial) {
    const int i = blockIdx.y, chunk = blockIdx.x, nchunks = gridDim.x;
    const long long per = (n + nchunks - 1) / nchunks;
    const long long b = chunk * per, e = min(n, b + per);
    double s = 0.0;
    for (long long x = b + threadIdx.x; x < e; x += blockDim.x) s = fma(V[i * ldv + x], y[x], s);
    s = block_sum(s);
    if (threadIdx.x == 0) partial[(long long)i * nchunks + chunk] = s;
}

__global__ void k_reduce_rows(const double* __restrict__ partial, int nchunks, double* __restrict__ out) {
    const int i = blockIdx.x;
    double s = 0.0;
    for (int c = threadIdx.x; c < nchunks; c += blockDim.x) s += partial[(long long)i * nchunks + c];
    s = block_sum(s);
    if (threadIdx.x == 0) out[i] = s;
}

__global__ void k_finite(const double* __restrict__ x, long long n, unsigned* err) {
    bool bad = false;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        if (!isfinite(x[i])) bad = true;
    if (bad) atomicOr(err, ERRBIT_NONFINITE);
}

// Lowest eigenpair of a small symmetric matrix (k <= 32) by cyclic Jacobi in FP64, one thread: the
// general form, for matrices whose lowest eigenvalues the FP32 basis of small_eig cannot tell apart.
// (a, v: shared memory -- as local arrays they would reserve 16 KB for every resident thread of the GPU)
__device__ __noinline__ void small_eig_serial(const double* G, int k, int ldg, double* yth, double (*a)[33],
                                              double (*v)[33]) {
    for (int i = 0; i < k; ++i)
        for (int j = 0; j < k; ++j) {
            a[i][j] = 0.5 * (G[i * ldg + j] + G[j * ldg + i]);
            v[i][j] = (i == j) ? 1.0 : 0.0;
        }
    for (int sweep = 0; sweep < 60; ++sweep) {
        double off = 0.0, dia = 0.0;
        for (int i = 0; i < k; ++i) {
            dia += a[i][i] * a[i][i];
            for (int j = i + 1; j < k; ++j) off += a[i][j] * a[i][j];
        }
        if (off <= 1e-34 * dia || off == 0.0) break;
        for (int p = 0; p < k; ++p)
            for (int q = p + 1; q < k; ++q) {
                double apq = a[p][q];
                if (apq == 0.0) continue;
                double zeta = (a[q][q] - a[p][p]) / (2.0 * apq);
                double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
                for (int r = 0; r < k; ++r) {
                    double arp = a[r][p], arq = a[r][q];
                    a[r][p] = c * arp - s * arq;
                    a[r][q] = s * arp + c * arq;
                }
                for (int r = 0; r < k; ++r) {
                    double apr = a[p][r], aqr = a[q][r];
                    a[p][r] = c * apr - s * aqr;
                    a[q][r] = s * apr + c * aqr;
                }
                for (int r = 0; r < k; ++r) {
                    double vrp = v[r][p], vrq = v[r][q];
                    v[r][p] = c * vrp - s * vrq;
                    v[r][q] = s * vrp + c * vrq;
                }
            }
    }
    int best = 0;
    for (int i = 1; i < k; ++i)
        if (a[i][i] < a[best][best]) best = i;
    yth[0] = a[best][best];
    for (int i = 0; i < k; ++i) yth[1 + i] = v[i][best];
}

// Lowest eigenpair (theta, y) of a small symmetric matrix G (k <= 32), one warp.
// The matrix is tiny, so dependent FP64 instructions (each tens of clocks here, a division or root a
// thousand) are the whole cost of an FP64 Jacobi: about 300 us at k = 4-8 on one thread.  Instead a
// parallel Jacobi in FP32 (round-robin pairs, on the matrix scaled by a power of two) gives an
// approximate eigenbasis Q, and the lowest pair is refined in FP64: theta = y.Gy, r = Gy - theta y,
// y <- y - sum_m q_m (q_m.r) / (lambda_m - theta), the sum in FP32 since it only has to be right to a
// few digits.  The residual falls by ~1e-6 a pass; passes go on while it falls, to eps |G|_F / 4, and the
// pair is accepted at |r| <= 4 eps |G|_F, else -- a cluster at the bottom, or non-finite entries -- the
// serial form runs.  Against 128 bits, 400 matrices each of k = 1..32 (random, dominant diagonal, arrow, near-
// degenerate, graded): |r| up to 0.7 eps |G|_F where the serial form has 4.1 (random), theta to 2 eps |G|_F and
// |y| to eps where it has 15 and 23.  One call at k = 4-8, cold caches: 300 -> about 18 us.
__device__ void small_eig(const double* G, int k, int ldg, double* yth) {
    constexpr unsigned ALL = 0xffffffffu;
    __shared__ double A[32][33], S[32][33];
    __shared__ float F[32][33], Q[32][33], cs[16], sn[16], rf[32], wf[32];
    __shared__ double ys[32];
    const int lane = threadIdx.x & 31;
    double amax = 0.0, fro = 0.0;
    for (int i = 0; i < k; ++i)
        if (lane < k) {
            const double x = 0.5 * (G[i * ldg + lane] + G[lane * ldg + i]);
            A[i][lane] = x;
            amax = fmax(amax, fabs(x));
        }
    for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(ALL, amax, o));
    bool ok = amax > 0.0 && amax < 1e300;
    int ex = 0;
    if (ok) frexp(amax, &ex);
    const double sc = ok ? ldexp(1.0, -ex) : 1.0;
    ok = ok && ex > -900;
    if (ok) {
        for (int i = 0; i < k; ++i)
            if (lane < k) {
                const double x = A[i][lane] * sc;
                A[i][lane] = x;
                F[i][lane] = (float)x;
                Q[i][lane] = i == lane ? 1.f : 0.f;
                fro = fma(x, x, fro);
            }
        fro = sqrt(warp_sum(fro));
        ok = fro < 1e300;                                  // false for NaN
    }
    __syncwarp();
    double y = 0.0, theta = 0.0;
    if (ok) {
        const int kp = k + (k & 1), np = kp / 2;
        // this lane's first 2 x 2 block (bi, bj) of F and first column pair rb of row rr of Q; 32 on,
        // both move by the same step
        const int bi0 = lane / np, bj0 = lane - bi0 * np, di = 32 / np, dj = 32 - di * np;
        for (int sweep = 0; sweep < 12 && k > 1; ++sweep) {
            float off = 0.f, dia = 0.f;
            for (int i = 0; i < k; ++i)
                if (lane < k) {
                    const float x = F[i][lane];
                    if (i == lane) dia = fmaf(x, x, dia);
                    else off = fmaf(x, x, off);
                }
            for (int o = 16; o > 0; o >>= 1) {
                off += __shfl_xor_sync(ALL, off, o);
                dia += __shfl_xor_sync(ALL, dia, o);
            }
            if (off <= 1e-13f * dia) break;
            for (int round = 0; round < kp - 1; ++round) {
                auto player = [&](int pos) {       // pos - 1 + round modulo kp - 1, plus 1; 0 stays
                    const int x = pos + round;
                    return pos == 0 ? 0 : (x > kp - 1 ? x - (kp - 1) : x);
                };
                if (lane < np) {
                    const int p = player(lane), q = player(kp - 1 - lane);
                    float c = 1.f, s = 0.f;
                    if (p < k && q < k) {
                        // cos 2t = |d| / sqrt(d^2 + h^2), c^2 = (1 + cos 2t) / 2: two reciprocal roots
                        // (entries are at most 1; below 1e-18 nothing is left to turn, or to underflow)
                        const float h = 2.f * F[p][q], d = F[q][q] - F[p][p];
                        if (fabsf(h) > 1e-18f) {
                            const float r = rsqrtf(fmaf(d, d, h * h));
                            const float i = rsqrtf(fmaf(0.5f * fabsf(d), r, 0.5f));
                            c = fmaf(0.5f * fabsf(d), r, 0.5f) * i;
                            s = (d >= 0.f ? 0.5f : -0.5f) * h * r * i;
                        }
                    }
                    cs[lane] = c;
                    sn[lane] = s;
                }
                __syncwarp();
                // (bj < np, so one carry a step) 2 x 2 blocks: they partition F
                for (int bi = bi0, bj = bj0; bi < np;) {
                    const int p0 = player(bi), q0 = player(kp - 1 - bi), p1 = player(bj), q1 = player(kp - 1 - bj);
                    const float ci = cs[bi], si = sn[bi], cj = cs[bj], sj = sn[bj];
                    const float a = p0 < k && p1 < k ? F[p0][p1] : 0.f, b = p0 < k && q1 < k ? F[p0][q1] : 0.f;
                    const float c = q0 < k && p1 < k ? F[q0][p1] : 0.f, d = q0 < k && q1 < k ? F[q0][q1] : 0.f;
                    const float a1 = cj * a - sj * b, b1 = sj * a + cj * b, c1 = cj * c - sj * d, d1 = sj * c + cj * d;
                    if (p0 < k && p1 < k) F[p0][p1] = ci * a1 - si * c1;
                    if (q0 < k && p1 < k) F[q0][p1] = si * a1 + ci * c1;
                    if (p0 < k && q1 < k) F[p0][q1] = ci * b1 - si * d1;
                    if (q0 < k && q1 < k) F[q0][q1] = si * b1 + ci * d1;
                    bi += di;
                    bj += dj;
                    if (bj >= np) {
                        bj -= np;
                        ++bi;
                    }
                }
                for (int r = bi0, b = bj0; r < k;) {
                    const int p = player(b), q = player(kp - 1 - b);
                    if (p < k && q < k) {
                        const float x = Q[r][p], z = Q[r][q];
                        Q[r][p] = cs[b] * x - sn[b] * z;
                        Q[r][q] = sn[b] * x + cs[b] * z;
                    }
                    r += di;
                    b += dj;
                    if (b >= np) {
                        b -= np;
                        ++r;
                    }
                }
                __syncwarp();
            }
        }
        int best = 0;
        for (int i = 1; i < k; ++i)
            if (F[i][i] < F[best][best]) best = i;
        const float lam0 = F[best][best];
        float inv = 0.f;                                       // 1 / (lambda_lane - lambda_best)
        bool apart = true;
        if (lane < k && lane != best) {
            apart = F[lane][lane] - lam0 > 4e-6f;
            inv = 1.f / fmaxf(F[lane][lane] - lam0, 4e-6f);
        }
        const bool isolated = __all_sync(ALL, apart);
        y = lane < k ? (double)Q[lane][best] : 0.0;
        y /= sqrt(warp_sum(y * y));
        double last = 1e300;
        for (int it = 0; it < 8; ++it) {
            ys[lane] = y;
            __syncwarp();
            double z0 = 0.0, z1 = 0.0;
            if (lane < k) {
                int j = 0;
                for (; j + 1 < k; j += 2) {
                    z0 = fma(A[j][lane], ys[j], z0);
                    z1 = fma(A[j + 1][lane], ys[j + 1], z1);
                }
                if (j < k) z0 = fma(A[j][lane], ys[j], z0);
            }
            z0 += z1;
            theta = warp_sum(y * z0);
            const double r = fma(-theta, y, z0);
            const double rn = warp_sum(r * r);
            // done when the residual no longer falls (squared: by less than 4) or is below rounding
            const double eps = 2.220446049250313e-16 * fro;
            if (!(rn > 0.0625 * eps * eps) || !(rn < 0.25 * last)) {
                ok = isolated && rn <= 16.0 * eps * eps;
                break;
            }
            last = rn;
            rf[lane] = (float)r;
            __syncwarp();
            float t = 0.f;
            if (lane < k)
                for (int i = 0; i < k; ++i) t = fmaf(Q[i][lane], rf[i], t);
            wf[lane] = -t * inv;
            __syncwarp();
            float dy = 0.f;
            if (lane < k)
                for (int m = 0; m < k; ++m) dy = fmaf(Q[lane][m], wf[m], dy);
            y += (double)dy;
            y *= fma(-0.5, warp_sum(y * y), 1.5);              // |y| is 1 to the correction squared
            if (it == 7) ok = false;
        }
    }
    if (!ok) {
        __syncwarp();
        if (lane == 0) small_eig_serial(G, k, ldg, yth, A, S);
        return;
    }
    if (lane == 0) yth[0] = ldexp(theta, ex);
    if (lane < k) yth[1 + lane] = y;
}

// ------------------------------------------------------------------------------------------
// Davidson's vector work between two matvecs, six launches (FP64, deterministic).
// Up to a few 10^4 elements these are launches of a few microseconds whose cost is the chain of them:
// as single operations -- dots, row sums, place, eigenpair, Ritz, row sums, preconditioner, two
// Gram-Schmidt passes of three, norm, scale: 18 launches and three host waits, 120 us a step with cold
// caches against 60 here (chain m = 64; FP64 sweep over 16 sites 147 -> 115 ms).  Each launch ends in a
// sum over all elements, and the CTA that arrives last adds up the CTAs' partial sums (in a fixed
// order) and does what follows on k numbers.
// Above, memory bounds them: V is read once a launch (three times in the correction, four before).
// A CTA has 128 threads: the FP64 units take a warp instruction every 64 clocks a scheduler, so few
// elements a CTA and a transposed warp reduction (9 additions for 8 sums instead of 40).
// ------------------------------------------------------------------------------------------
constexpr int DAV_THREADS = 128, DAV_GROUP = 8;

// Sum of v[j] over the CTA in thread j < 8 (any value in others).
__device__ __forceinline__ double dav_cta_sum(double (&v)[DAV_GROUP]) {
    constexpr unsigned ALL = 0xffffffffu;
    __shared__ double red[DAV_THREADS / 32][DAV_GROUP];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int h = DAV_GROUP / 2, o = 16; h >= 1; h /= 2, o /= 2)       // halve the sums, double the lanes
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const bool up = lane & o;
            v[j] = (up ? v[j + h] : v[j]) + __shfl_xor_sync(ALL, up ? v[j] : v[j + h], o);
        }
    v[0] += __shfl_xor_sync(ALL, v[0], 2);
    v[0] += __shfl_xor_sync(ALL, v[0], 1);
    __syncthreads();                                                   // red's last readers
    if ((lane & 3) == 0) red[w][lane >> 2] = v[0];                     // bits 16, 8, 4 of the lane: j's bits
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < DAV_GROUP)
        s = (red[0][threadIdx.x] + red[1][threadIdx.x]) + (red[2][threadIdx.x] + red[3][threadIdx.x]);
    return s;
}
// True in every thread of the CTA that arrives last (with every CTA's earlier writes visible);
// *ctr is zero before and after a launch.
__device__ __forceinline__ bool dav_last(unsigned* ctr) {
    __shared__ unsigned last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ctr, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    if (threadIdx.x == 0) *ctr = 0u;
    __threadfence();
    return true;
}
// Sum of a row of partial sums, one warp.
__device__ __forceinline__ double dav_row(const double* partial, int row) {
    const double* p = partial + (long long)row * gridDim.x;
    double s = 0.0;
    for (int c = threadIdx.x & 31; c < gridDim.x; c += 32) s += __ldcg(p + c);
    return warp_sum(s);
}
#define DAV_FOR(x) \
    for (long long x = (long long)blockIdx.x * DAV_THREADS + threadIdx.x; x < n; x += (long long)gridDim.x * DAV_THREADS)

// G's new column k (V_i . AV_k, i <= k) and row (V_k . AV_i, i < k); eig: then the lowest pair of the
// (k + 1) x (k + 1) matrix into yth (theta, coefficients).
__global__ void __launch_bounds__(DAV_THREADS) k_dav_gram(const double* __restrict__ V, const double* __restrict__ AV,
                                                          long long n, int k, int ldg, double* G, double* partial,
                                                          unsigned* ctr, int eig, double* yth) {
    const double* vk = V + k * n;
    const double* ak = AV + k * n;
    for (int i0 = 0; i0 <= k; i0 += DAV_GROUP / 2) {
        double acc[DAV_GROUP] = {};
        DAV_FOR(x) {
            const double a = ak[x], v = vk[x];
#pragma unroll
            for (int j = 0; j < DAV_GROUP / 2; ++j) {
                const long long o = (i0 + j) * n + x;
                if (i0 + j <= k) acc[j] = fma(V[o], a, acc[j]);
                if (i0 + j < k) acc[DAV_GROUP / 2 + j] = fma(AV[o], v, acc[DAV_GROUP / 2 + j]);
            }
        }
        const double s = dav_cta_sum(acc);
        const int j = threadIdx.x & (DAV_GROUP / 2 - 1);
        if (threadIdx.x < DAV_GROUP && i0 + j <= k)
            partial[(long long)(threadIdx.x < DAV_GROUP / 2 ? i0 + j : ldg + i0 + j) * gridDim.x + blockIdx.x] = s;
    }
    if (!dav_last(ctr)) return;
    for (int i = threadIdx.x >> 5; i <= 2 * k; i += DAV_THREADS / 32) {     // k + 1 of the column, k of the row
        const double s = dav_row(partial, i <= k ? i : ldg + i - k - 1);
        if ((threadIdx.x & 31) == 0) G[i <= k ? (long long)i * ldg + k : (long long)k * ldg + i - k - 1] = s;
    }
    __syncthreads();
    if (eig && threadIdx.x < 32) small_eig(G, k + 1, ldg, yth);
}

// u = V y, Au = AV y, r = Au - theta u; norms[0] = |r|^2, norms[1] = |u|^2; host[0..2] = |r|^2, |u|^2, theta
// (pinned memory that the host reads after an event; as copies in the stream, three an iteration: 16-site
// FP64 sweep at m = 64 96.3 ms, 89.7 this way; four bf16 regions at m = 128 83.7, 79.8).
__global__ void __launch_bounds__(DAV_THREADS) k_dav_ritz(const double* __restrict__ V, const double* __restrict__ AV,
                                                          long long n, int k, const double* __restrict__ yth,
                                                          double* __restrict__ u, double* __restrict__ Au,
                                                          double* __restrict__ r, double* partial, unsigned* ctr,
                                                          double* __restrict__ norms, double* __restrict__ host) {
    __shared__ double y[33];
    if (threadIdx.x <= k) y[threadIdx.x] = yth[threadIdx.x];
    __syncthreads();
    double acc[DAV_GROUP] = {};
    DAV_FOR(x) {
        double uu = 0.0, aa = 0.0;
#pragma unroll 4
        for (int i = 0; i < k; ++i) {
            uu = fma(y[1 + i], V[i * n + x], uu);
            aa = fma(y[1 + i], AV[i * n + x], aa);
        }
        const double rr = aa - y[0] * uu;
        u[x] = uu;
        Au[x] = aa;
        r[x] = rr;
        acc[0] = fma(rr, rr, acc[0]);
        acc[1] = fma(uu, uu, acc[1]);
    }
    const double s = dav_cta_sum(acc);
    if (threadIdx.x < 2) partial[(long long)threadIdx.x * gridDim.x + blockIdx.x] = s;
    if (!dav_last(ctr)) return;
    if (threadIdx.x < 64) {
        const double t = dav_row(partial, threadIdx.x >> 5);
        if ((threadIdx.x & 31) == 0) norms[threadIdx.x >> 5] = host[threadIdx.x >> 5] = t;
    }
    if (threadIdx.x == 64) host[2] = y[0];
}

// Gram-Schmidt of the correction t against V_0 .. V_{k-1}, one pass per launch.  FIRST: t = r / (theta -
// diag) (the denominator at least fl in size); else t -= V c.  Then c_out = V^T t.
template <bool FIRST>
__global__ void __launch_bounds__(DAV_THREADS) k_dav_correct(const double* __restrict__ V, long long n, int k,
                                                             const double* __restrict__ r,
                                                             const double* __restrict__ diag,
                                                             const double* __restrict__ theta, double fl,
                                                             const double* __restrict__ c, double* t, double* partial,
                                                             unsigned* ctr, double* __restrict__ c_out) {
    __shared__ double cs[32];
    if (!FIRST && threadIdx.x < k) cs[threadIdx.x] = c[threadIdx.x];
    __syncthreads();
    const double th = FIRST ? theta[0] : 0.0;
    for (int i0 = 0; i0 < k; i0 += DAV_GROUP) {
        const int g = min(DAV_GROUP, k - i0);
        double acc[DAV_GROUP] = {};
        DAV_FOR(x) {
            double v[DAV_GROUP], tx;
#pragma unroll
            for (int j = 0; j < DAV_GROUP; ++j) v[j] = j < g ? V[(i0 + j) * n + x] : 0.0;
            if (i0 == 0) {
                if (FIRST) {
                    double den = th - diag[x];
                    if (fabs(den) < fl) den = den >= 0.0 ? fl : -fl;
                    tx = r[x] / den;
                } else {
                    tx = t[x];
#pragma unroll
                    for (int j = 0; j < DAV_GROUP; ++j)
                        if (j < g) tx = fma(-cs[j], v[j], tx);
                    for (int i = DAV_GROUP; i < k; ++i) tx = fma(-cs[i], V[i * n + x], tx);
                }
                t[x] = tx;
            } else {
                tx = t[x];                          // this thread's own write
            }
#pragma unroll
            for (int j = 0; j < DAV_GROUP; ++j)
                if (j < g) acc[j] = fma(v[j], tx, acc[j]);
        }
        const double s = dav_cta_sum(acc);
        if (threadIdx.x < g) partial[(long long)(i0 + threadIdx.x) * gridDim.x + blockIdx.x] = s;
    }
    if (!dav_last(ctr)) return;
    for (int i = threadIdx.x >> 5; i < k; i += DAV_THREADS / 32) {
        const double s = dav_row(partial, i);
        if ((threadIdx.x & 31) == 0) c_out[i] = s;
    }
}

// t -= V c (k vectors; none: t is left), *nrm2 = *host = |t|^2 (host: pinned memory or null).
__global__ void __launch_bounds__(DAV_THREADS) k_dav_norm(const double* __restrict__ V, long long n, int k,
                                                          const double* __restrict__ c, double* t, double* partial,
                                                          unsigned* ctr, double* __restrict__ nrm2,
                                                          double* __restrict__ host) {
    __shared__ double cs[32];
    if (threadIdx.x < k) cs[threadIdx.x] = c[threadIdx.x];
    __syncthreads();
    double acc[DAV_GROUP] = {};
    DAV_FOR(x) {
        double tx = t[x];
#pragma unroll 8
        for (int i = 0; i < k; ++i) tx = fma(-cs[i], V[i * n + x], tx);
        if (k > 0) t[x] = tx;
        acc[0] = fma(tx, tx, acc[0]);
    }
    const double s = dav_cta_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
    if (!dav_last(ctr)) return;
    if (threadIdx.x < 32) {
        const double v = dav_row(partial, 0);
        if (threadIdx.x == 0) {
            *nrm2 = v;
            if (host) *host = v;
        }
    }
}

// y = x / sqrt(*nrm2); zero where that root is below `floor_` (the caller stops there).
__global__ void __launch_bounds__(256) k_dav_unit(const double* __restrict__ x, const double* __restrict__ nrm2,
                                                  double floor_, long long n, double* __restrict__ y) {
    const double root = sqrt(nrm2[0]);
    const double s = root < floor_ ? 0.0 : 1.0 / root;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = s == 0.0 ? 0.0 : x[i] * s;
}

// ------------------------------------------------------------------------------------------
// One-sided Jacobi SVD (Hestenes).  W holds the sector matrix column-major (p x n, n <= p); pairs
// of columns are rotated until mutually orthogonal; V accumulates the rotations.  The rounds of
// a sweep follow the round-robin tournament (n/2 disjoint pairs per round, n-1 rounds).
// ------------------------------------------------------------------------------------------
template <class T>
__global__ void k_svd_init_v(const SvdSec* __restrict__ secs, T* __restrict__ V) {
    const SvdSec s = secs[blockIdx.y];
    const long long total = (long long)s.n * s.n;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        int c = (int)(e / s.n), r = (int)(e % s.n);
        V[s.v_off + e] = (r == c) ? T(1) : T(0);
    }
}

// Round-robin pairing: position 0 fixed, positions 1..npad-1 rotate by `round`.
__device__ __forceinline__ int rr_player(int pos, int round, int npad) {
    return pos == 0 ? 0 : ((pos - 1 + round) % (npad - 1)) + 1;
}

template <class T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One warp rotates one column pair; returns true if it rotated.  Each lane keeps its share of
// both columns (rows lane, lane+32, ...) in registers, so every phase costs one memory latency.
constexpr int JREG = 32;   // register-resident rows per lane: p and n up to 32*32 = 1024
template <class T>
__device__ __forceinline__ bool jacobi_pair(const SvdSec& s, int pi, int round, T* __restrict__ W,
                                            T* __restrict__ V, T tol, T floor_, int lane) {
    if (round >= s.npad - 1) return false;
    int i = rr_player(pi, round, s.npad);
    int j = rr_player(s.npad - 1 - pi, round, s.npad);
    if (i > j) { int t = i; i = j; j = t; }
    if (j >= s.n) return false;                      // bye against the padding column
    T* ci = W + s.w_off + (long long)i * s.p;
    T* cj = W + s.w_off + (long long)j * s.p;
    T* vi = V + s.v_off + (long long)i * s.n;
    T* vj = V + s.v_off + (long long)j * s.n;
    T al = 0, be = 0, ga = 0;
    if (s.p <= 32 * JREG && s.n <= 32 * JREG) {
        T x[JREG], y[JREG];
#pragma unroll
        for (int k = 0; k < JREG; ++k) {
            const int r = lane + 32 * k;
            x[k] = r < s.p ? ci[r] : T(0);
            y[k] = r < s.p ? cj[r] : T(0);
        }
#pragma unroll
        for (int k = 0; k < JREG; ++k) {
            al = fma(x[k], x[k], al);
            be = fma(y[k], y[k], be);
            ga = fma(x[k], y[k], ga);
        }
        al = wsum(al);
        be = wsum(be);
        ga = wsum(ga);
        if (ga == T(0) || !(fabs(ga) > tol * sqrt(al * be)) || fmin(al, be) <= floor_) return false;
        T zeta = (be - al) / (T(2) * ga);
        T t = (zeta >= T(0) ? T(1) : T(-1)) / (fabs(zeta) + sqrt(T(1) + zeta * zeta));
        T c = T(1) / sqrt(T(1) + t * t), sn = c * t;
        T u[JREG], w[JREG];
#pragma unroll
        for (int k = 0; k < JREG; ++k) {
            const int r = lane + 32 * k;
            u[k] = r < s.n ? vi[r] : T(0);
            w[k] = r < s.n ? vj[r] : T(0);
        }
#pragma unroll
        for (int k = 0; k < JREG; ++k) {
            const int r = lane + 32 * k;
            if (r < s.p) {
                ci[r] = c * x[k] - sn * y[k];
                cj[r] = sn * x[k] + c * y[k];
            }
            if (r < s.n) {
                vi[r] = c * u[k] - sn * w[k];
                vj[r] = sn * u[k] + c * w[k];
            }
        }
        return true;
    }
    for (int r = lane; r < s.p; r += 32) {
        T x = ci[r], y = cj[r];
        al = fma(x, x, al);
        be = fma(y, y, be);
        ga = fma(x, y, ga);
    }
    al = wsum(al);
    be = wsum(be);
    ga = wsum(ga);
    if (ga == T(0) || !(fabs(ga) > tol * sqrt(al * be)) || fmin(al, be) <= floor_) return false;
    T zeta = (be - al) / (T(2) * ga);
    T t = (zeta >= T(0) ? T(1) : T(-1)) / (fabs(zeta) + sqrt(T(1) + zeta * zeta));
    T c = T(1) / sqrt(T(1) + t * t), sn = c * t;
    for (int r = lane; r < s.p; r += 32) {
        T x = ci[r], y = cj[r];
        ci[r] = c * x - sn * y;
        cj[r] = sn * x + c * y;
    }
    for (int r = lane; r < s.n; r += 32) {
        T x = vi[r], y = vj[r];
        vi[r] = c * x - sn * y;
        vj[r] = sn * x + c * y;
    }
    return true;
}

// All sweeps of all sectors in one cooperative launch; bounded grid barrier between rounds.
// rot[sweep] counts the warps that rotated in that sweep (zeroed by the host); *sweeps = sweeps
// run; bar: 3 zeroed words for the barrier.
template <class T>
__global__ void k_jacobi_coop(const SvdSec* __restrict__ secs, const int* __restrict__ pair_sec, int npairs,
                              int maxnpad, int max_sweeps, T* __restrict__ W, T* __restrict__ V, T tol,
                              const double* __restrict__ floor2, int* __restrict__ rot, int* __restrict__ sweeps,
                              unsigned* __restrict__ bar, unsigned* __restrict__ err) {
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    int sweep = 0;
    bool alive = true;
    for (; sweep < max_sweeps && alive; ++sweep) {
        int mine = 0;
        for (int round = 0; round < maxnpad - 1 && alive; ++round) {
            for (int w = gw; w < npairs; w += nw) {
                const int si = pair_sec[w];
                const SvdSec s = secs[si];
                if (jacobi_pair<T>(s, w - s.pair0, round, W, V, tol * sqrt((T)s.p), floor2 ? (T)floor2[si] : T(0), lane)) mine = 1;
            }
            alive = grid_barrier(bar, gridDim.x, err);
        }
        if (!alive) break;
        if (lane == 0 && mine) atomicAdd(&rot[sweep], 1);
        alive = grid_barrier(bar, gridDim.x, err);
        if (!alive) break;
        if (*((volatile int*)&rot[sweep]) == 0) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *sweeps = sweep + 1;
}

// One round of one sweep of the scalar Jacobi (one warp per pair); rot[sweep] set when a pair
// rotated.  A launch whose previous sweep rotated nothing returns at once.
template <class T>
__global__ void k_jacobi_round(const SvdSec* __restrict__ secs, const int* __restrict__ pair_sec, int npairs,
                               int round, int sweep, T* __restrict__ W, T* __restrict__ V, T tol,
                               const double* __restrict__ floor2, int* __restrict__ rot) {
    if (sweep > 0 && *((volatile int*)&rot[sweep - 1]) == 0) return;
    const int lane = threadIdx.x & 31;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= npairs) return;
    const int si = pair_sec[w];
    const SvdSec s = secs[si];
    if (jacobi_pair<T>(s, w - s.pair0, round, W, V, tol * sqrt((T)s.p), floor2 ? (T)floor2[si] : T(0), lane) && lane == 0)
        rot[sweep] = 1;
}

// floor2[s] = (eta * |W_s|_F)^2: columns below it are left unrotated (below working precision).
template <class T>
__global__ void k_svd_floor(const SvdSec* __restrict__ secs, const T* __restrict__ W, double eta,
                            double* __restrict__ floor2) {
    const SvdSec s = secs[blockIdx.x];
    double a = 0.0;
    const long long total = (long long)s.p * s.n;
    for (long long e = threadIdx.x; e < total; e += blockDim.x) {
        double x = (double)W[s.w_off + e];
        a = fma(x, x, a);
    }
    a = block_sum(a);
    if (threadIdx.x == 0) floor2[blockIdx.x] = eta * eta * a;
}

// sig[s_off + i] = |W_i| (FP64): one warp per column.
template <class T>
__global__ void k_svd_norms(const SvdSec* __restrict__ secs, const T* __restrict__ W, double* __restrict__ sig) {
    const SvdSec s = secs[blockIdx.y];
    const int lane = threadIdx.x & 31, c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (c >= s.n) return;
    const T* col = W + s.w_off + (long long)c * s.p;
    double a = 0.0, b = 0.0;
    int r = lane;
    for (; r + 32 < s.p; r += 64) {
        const double x = (double)col[r], y = (double)col[r + 32];
        a = fma(x, x, a);
        b = fma(y, y, b);
    }
    if (r < s.p) a = fma((double)col[r], (double)col[r], a);
    a = warp_sum(a + b);
    if (lane == 0) sig[s.s_off + c] = sqrt(a);
}

// Norms are not negative, so they order like their bit patterns (integer comparisons: a double's
// would run on the FP64 pipe).
__device__ __forceinline__ long long norm_bits(double x) { return __double_as_longlong(x); }

// order[s_off + r] = column with the r-th largest norm (ties: lower index): one warp per column.  (One
// CTA per sector did norms and ranks before: 600 us for the 68 sectors of four m = 2000 bonds, 20 now.)
__global__ void k_svd_order(const SvdSec* __restrict__ secs, const double* __restrict__ sig, int* __restrict__ order) {
    const SvdSec s = secs[blockIdx.y];
    const int lane = threadIdx.x & 31, c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (c >= s.n) return;
    const long long v = norm_bits(sig[s.s_off + c]);
    int rank = 0;
    for (int o = lane; o < s.n; o += 32) {
        const long long w = norm_bits(sig[s.s_off + o]);
        rank += (w > v) || (w == v && o < c);
    }
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane == 0) order[s.s_off + rank] = c;
}

// ------------------------------------------------------------------------------------------
// Truncation selection.  Keys (lambda desc, sector asc, position asc) over all sectors' values.
//   k_trunc_flat   flat arrays lam[g], sec[g] (sector order, descending inside)
//   k_trunc_rank   rank of every candidate (lambda > rel_cutoff * lambda_max) among candidates
//   k_trunc_count  kept[s] and weights: total sum lambda^2, kept sum lambda^2
// ------------------------------------------------------------------------------------------
__global__ void k_trunc_flat(const SvdSec* __restrict__ secs, int nsec, const double* __restrict__ sig,
                             const int* __restrict__ order, double* __restrict__ lam, int* __restrict__ sec,
                             double* __restrict__ lmax) {
    const int s = blockIdx.x;
    const SvdSec S = secs[s];
    double mx = 0.0;
    for (int i = threadIdx.x; i < S.n; i += blockDim.x) {
        double v = sig[S.s_off + order[S.s_off + i]];
        lam[S.s_off + i] = v;
        sec[S.s_off + i] = s;
        mx = fmax(mx, v);
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __shared__ double red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, red[w]);
        lmax[s] = m;
    }
}

// One warp per value; the flat index orders like (sector, position), so it breaks ties.  (A thread per
// value and double comparisons before: 580 us for the 4000 values of an m = 2000 bond, 20 now.)
__global__ void k_trunc_rank(const double* __restrict__ lam, int total, const double* __restrict__ lmax_sec, int nsec,
                             double rel_cutoff, int* __restrict__ rank) {
    const int lane = threadIdx.x & 31, g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= total) return;
    double m = 0.0;
    for (int s = lane; s < nsec; s += 32) m = fmax(m, lmax_sec[s]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    const double thr = rel_cutoff * m, v = lam[g];
    int r = -1;
    if (v > thr) {                                   // the same in every lane
        const long long tb = norm_bits(thr), vb = norm_bits(v), inf = 0x7FF0000000000000ll;
        r = 0;
        for (int o = lane; o < total; o += 32) {
            const long long w = norm_bits(lam[o]);
            r += w > tb && w <= inf && (w > vb || (w == vb && o < g));
        }
        r = __reduce_add_sync(0xffffffffu, r);
    }
    if (lane == 0) rank[g] = r;
}

__global__ void __launch_bounds__(1024) k_trunc_count(const double* __restrict__ lam, const int* __restrict__ sec,
                                                      const int* __restrict__ rank, int total, int nsec, int m_max,
                                                      double degen_tol, int* __restrict__ kept,
                                                      double* __restrict__ weights) {
    __shared__ double s_next;
    __shared__ int s_cnt[256];
    if (threadIdx.x == 0) s_next = -1.0;
    for (int s = threadIdx.x; s < 256; s += blockDim.x) s_cnt[s] = 0;
    __syncthreads();
    double tot = 0.0;
    for (int g = threadIdx.x; g < total; g += blockDim.x) {
        tot += lam[g] * lam[g];
        if (rank[g] == m_max) s_next = lam[g];
    }
    tot = block_sum(tot);
    const double nxt = s_next;
    double kw = 0.0;
    for (int g = threadIdx.x; g < total; g += blockDim.x) {
        const int r = rank[g];
        const double a = lam[g];
        if (r >= 0 && r < m_max && (nxt < 0.0 || a > nxt * (1.0 + degen_tol))) {
            kw += a * a;
            atomicAdd(&s_cnt[sec[g]], 1);
        }
    }
    kw = block_sum(kw);
    for (int s = threadIdx.x; s < nsec; s += blockDim.x) kept[s] = s_cnt[s];
    if (threadIdx.x == 0) {
        weights[0] = tot;
        weights[1] = kw;
    }
}

inline int grid_for(long long elems, int cap = 4096) {
    long long g = (elems + 255) / 256;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

}  // namespace

// ------------------------------------------------------------------------------------------
// Launch wrappers
// ------------------------------------------------------------------------------------------
void launch_gemm_f32(const GProb* probs, const GSeg* segs, const GTile* tiles, int ntiles, const float* A, const float* B,
                     float* C, cudaStream_t st) {
    if (ntiles <= 0) return;
    k_gemm_f32<<<ntiles, 64, 0, st>>>(probs, segs, tiles, A, B, C);
    PD_LAUNCHED();
}

F64Shape f64_shape(const std::vector<GProb>& probs, const std::vector<GSeg>& segs) {
    // 16 x 16 tiles and their mean K decide.  A tile's chain is 8 K warp instructions of 64 clocks on
    // one scheduler, and the 4 kSMs schedulers want several tiles each: with 16 or more (or a K too
    // short to divide) a warp takes a tile alone, else four warps share one; eight where there are no
    // more tiles than schedulers and K is at least 128, sixteen where there are no more than SMs and K is
    // at least 256.  Measured, one / four / eight / sixteen warps a tile, in us:
    //   5000 of 15x15x15 (5000 tiles)          76 /   89 /  199 /  342   (64 x 64 CTA tiles before: 541)
    //    400 of 150x150x150 (40000)          2300 / 2476 / 3563 / 4583   (3859)
    //     17 of 320x320x640 (6800)           1960 / 1868 / 2121 / 2297   (1957; 1.19 TFLOP/s of the 1.25 measured peak)
    //     34 of 80x80x80 (850)                 65 /   47 /   70 /   94   (98)
    //    320x320x640 (400)                    227 /  139 /  147 /  158
    //     10 of 100x100x128 (490)              80 /   45 /   55 /   70
    //    160x160x640 (100)                    226 /   64 /   54 /   58
    //     52 of 15x15, 98 x K = 15 (52)       465 /  130 /  108 /  108   (1625)
    // Below one tile an SM eight and sixteen win over four by a sixth; the line of the eight-warp shape was
    // drawn against sixteen (R stage of the m = 500 matvec 578 -> 440 us): from 153 to 608 tiles four does as
    // well or better (that call 1110 us with the rule, 1052 with four).
    long long tiles = 0, kt = 0;
    for (const GProb& p : probs) {
        const long long t = (long long)((p.M + 15) / 16) * ((p.N + 15) / 16);
        long long k = 0;
        for (int s = 0; s < p.nseg; ++s) k += segs[p.seg0 + s].K;
        tiles += t;
        kt += t * k;
    }
    const double kmean = tiles ? (double)kt / (double)tiles : 0.0;
    if (tiles >= 9728 || kmean < 16.0) return {32, 1};
    if (tiles <= kSMs && kmean >= 256.0) return {16, 16};
    if (tiles <= 4 * kSMs && kmean >= 128.0) return {16, 8};
    return {16, 4};
}

void launch_gemm_f64(const GProb* probs, const GSeg* segs, const GTile* tiles, int ntiles, int edge, F64Shape shape,
                     const double* A, const double* B, double* C, cudaStream_t st) {
    if (ntiles <= 0) return;
    const int side = edge / shape.tile;
    const long long grid = (long long)ntiles * side * side;
    PD_REQUIRE(side >= 1 && side * shape.tile == edge && grid < (1LL << 31), DMRG_ERR_CAPACITY, "FP64 GEMM tile list");
    if (shape.ksplit == 1) k_gemm_f64<1><<<(unsigned)grid, 128, 0, st>>>(probs, segs, tiles, side, A, B, C);
    else if (shape.ksplit == 4) k_gemm_f64<4><<<(unsigned)grid, 128, 0, st>>>(probs, segs, tiles, side, A, B, C);
    else if (shape.ksplit == 8) k_gemm_f64<8><<<(unsigned)grid, 256, 0, st>>>(probs, segs, tiles, side, A, B, C);
    else k_gemm_f64<16><<<(unsigned)grid, 512, 0, st>>>(probs, segs, tiles, side, A, B, C);
    PD_LAUNCHED();
}

template <class Tin, class Tout>
void launch_copy(const CopyJob* jobs, const int2* chunks, int nchunks, const Tin* src, Tout* dst, cudaStream_t st) {
    if (nchunks <= 0) return;
    k_copy<Tin, Tout><<<nchunks, 256, 0, st>>>(jobs, chunks, src, dst);
    PD_LAUNCHED();
}

template <class Tin, class Tout>
void launch_convert(const Tin* src, Tout* dst, long long n, cudaStream_t st) {
    if (n <= 0) return;
    k_convert<Tin, Tout><<<(unsigned)std::max<long long>(1, std::min<long long>((n + 2047) / 2048, 8 * kSMs)), 256, 0, st>>>(
        src, dst, n);
    PD_LAUNCHED();
}
template void launch_convert<double, float>(const double*, float*, long long, cudaStream_t);
template void launch_convert<double, __nv_bfloat16>(const double*, __nv_bfloat16*, long long, cudaStream_t);
template void launch_convert<float, double>(const float*, double*, long long, cudaStream_t);
template void launch_convert<float, __nv_bfloat16>(const float*, __nv_bfloat16*, long long, cudaStream_t);

template <class Tin, class Tout>
void launch_mix(const MixJob* jobs, const int2* chunks, int nchunks, const MixTerm* terms, const Tin* in,
                Tout* out, cudaStream_t st) {
    if (nchunks <= 0) return;
    k_mix<Tin, Tout><<<nchunks, 256, 0, st>>>(jobs, chunks, terms, in, out);
    PD_LAUNCHED();
}

template <class T>
void launch_diag(const DiagJob* jobs, const int2* chunks, int nchunks, const DiagTerm* terms, const T* Ls, int ldl,
                 const T* Rs, int ldr, double* out, cudaStream_t st) {
    if (nchunks <= 0) return;
    k_diag<T><<<nchunks, 256, 0, st>>>(jobs, chunks, terms, Ls, ldl, Rs, ldr, out);
    PD_LAUNCHED();
}

template void launch_copy<double, double>(const CopyJob*, const int2*, int, const double*, double*, cudaStream_t);
template void launch_copy<double, float>(const CopyJob*, const int2*, int, const double*, float*, cudaStream_t);
template void launch_copy<double, __nv_bfloat16>(const CopyJob*, const int2*, int, const double*, __nv_bfloat16*, cudaStream_t);
template void launch_copy<float, double>(const CopyJob*, const int2*, int, const float*, double*, cudaStream_t);
template void launch_copy<float, float>(const CopyJob*, const int2*, int, const float*, float*, cudaStream_t);
template void launch_copy<float, __nv_bfloat16>(const CopyJob*, const int2*, int, const float*, __nv_bfloat16*, cudaStream_t);
template void launch_mix<double, double>(const MixJob*, const int2*, int, const MixTerm*, const double*, double*, cudaStream_t);
template void launch_mix<float, float>(const MixJob*, const int2*, int, const MixTerm*, const float*, float*, cudaStream_t);
template void launch_mix<float, __nv_bfloat16>(const MixJob*, const int2*, int, const MixTerm*, const float*, __nv_bfloat16*, cudaStream_t);
template void launch_diag<double>(const DiagJob*, const int2*, int, const DiagTerm*, const double*, int, const double*, int, double*, cudaStream_t);
template void launch_diag<float>(const DiagJob*, const int2*, int, const DiagTerm*, const float*, int, const float*, int, double*, cudaStream_t);

void launch_dots(const double* V, long long ldv, int k, const double* y, long long n, double* partial,
                 int nchunks, double* out, cudaStream_t st) {
    if (k <= 0) return;
    k_dots_partial<<<dim3(nchunks, k), 256, 0, st>>>(V, ldv, y, n, partial);
    PD_LAUNCHED();
    k_reduce_rows<<<k, 256, 0, st>>>(partial, nchunks, out);
    PD_LAUNCHED();
}

int dav_grid(long long n) {
    return (int)std::max<long long>(1, std::min<long long>((n + DAV_THREADS - 1) / DAV_THREADS, 4 * kSMs));
}

void launch_dav_gram(const double* V, const double* AV, long long n, int k, int kmax, double* G, double* partial,
                     unsigned* ctr, bool eig, double* yth, cudaStream_t st) {
    PD_REQUIRE(k >= 0 && k < kmax && kmax <= 32, DMRG_ERR_CAPACITY, "Davidson subspace larger than 32");
    k_dav_gram<<<dav_grid(n), DAV_THREADS, 0, st>>>(V, AV, n, k, kmax, G, partial, ctr, eig ? 1 : 0, yth);
    PD_LAUNCHED();
}

void launch_dav_ritz(const double* V, const double* AV, long long n, int k, const double* yth, double* u, double* Au,
                     double* r, double* partial, unsigned* ctr, double* norms, double* host, cudaStream_t st) {
    k_dav_ritz<<<dav_grid(n), DAV_THREADS, 0, st>>>(V, AV, n, k, yth, u, Au, r, partial, ctr, norms, host);
    PD_LAUNCHED();
}

void launch_dav_correct(const double* V, long long n, int k, const double* r, const double* diag, const double* theta,
                        double fl, double* t, double* c1, double* c2, double* partial, unsigned* ctr, double* nrm2,
                        double* host, cudaStream_t st) {
    k_dav_correct<true><<<dav_grid(n), DAV_THREADS, 0, st>>>(V, n, k, r, diag, theta, fl, nullptr, t, partial, ctr, c1);
    PD_LAUNCHED();
    k_dav_correct<false>
        <<<dav_grid(n), DAV_THREADS, 0, st>>>(V, n, k, nullptr, nullptr, nullptr, 0.0, c1, t, partial, ctr, c2);
    PD_LAUNCHED();
    k_dav_norm<<<dav_grid(n), DAV_THREADS, 0, st>>>(V, n, k, c2, t, partial, ctr, nrm2, host);
    PD_LAUNCHED();
}

void launch_dav_norm(double* x, long long n, double* partial, unsigned* ctr, double* nrm2, cudaStream_t st) {
    k_dav_norm<<<dav_grid(n), DAV_THREADS, 0, st>>>(nullptr, n, 0, nullptr, x, partial, ctr, nrm2, nullptr);
    PD_LAUNCHED();
}

void launch_dav_unit(const double* x, const double* nrm2, double floor_, long long n, double* y, cudaStream_t st) {
    k_dav_unit<<<grid_for(n), 256, 0, st>>>(x, nrm2, floor_, n, y);
    PD_LAUNCHED();
}

void launch_finite_check(const double* x, long long n, unsigned* err, cudaStream_t st) {
    k_finite<<<grid_for(n, 1024), 256, 0, st>>>(x, n, err);
    PD_LAUNCHED();
}

template <class T>
void launch_svd_init_v(const SvdSec* secs, int nsec, int max_n, T* V, cudaStream_t st) {
    if (nsec <= 0) return;
    k_svd_init_v<T><<<dim3(grid_for((long long)max_n * max_n, 256), nsec), 256, 0, st>>>(secs, V);
    PD_LAUNCHED();
}
template void launch_svd_init_v<double>(const SvdSec*, int, int, double*, cudaStream_t);
template void launch_svd_init_v<float>(const SvdSec*, int, int, float*, cudaStream_t);

template <class T>
void launch_jacobi(const SvdSec* secs, int nsec, const int* pair_sec, int npairs, int maxnpad, int max_sweeps, T* W,
                   T* V, T tol, double eta, double* floor2, int* rot, int* sweeps, unsigned* bar, unsigned* err,
                   cudaStream_t st) {
    if (npairs <= 0 || maxnpad < 2) return;
    const double* fl = nullptr;
    if (eta > 0.0) {
        k_svd_floor<T><<<nsec, 256, 0, st>>>(secs, W, eta, floor2);
        PD_LAUNCHED();
        fl = floor2;
    }
    const int threads = 128;   // register-heavy pair updates: small blocks keep several per SM
    if (g_sm_cap > 0) {
        // regions run concurrently: one launch per round (no grid barrier spinning on SMs that
        // other regions' kernels need), convergence read one sweep behind
        const int grid = (npairs * 32 + threads - 1) / threads;
        int* hrot = sweep_flags_host(max_sweeps);
        std::vector<cudaEvent_t> evs(max_sweeps, nullptr);
        int done = max_sweeps;
        auto cleanup = [&]() {
            for (auto e : evs)
                if (e) cudaEventDestroy(e);
        };
        try {
            for (int sweep = 0; sweep < max_sweeps; ++sweep) {
                for (int round = 0; round < maxnpad - 1; ++round) {
                    k_jacobi_round<T><<<grid, threads, 0, st>>>(secs, pair_sec, npairs, round, sweep, W, V, tol, fl,
                                                                rot);
                    PD_LAUNCHED();
                }
                PD_CK(cudaMemcpyAsync(hrot + sweep, rot + sweep, sizeof(int), cudaMemcpyDeviceToHost, st));
                PD_CK(cudaEventCreateWithFlags(&evs[sweep], cudaEventDisableTiming));
                PD_CK(cudaEventRecord(evs[sweep], st));
                if (sweep > 0) {
                    PD_CK(cudaEventSynchronize(evs[sweep - 1]));
                    if (hrot[sweep - 1] == 0) {
                        done = sweep;
                        break;
                    }
                }
            }
        } catch (...) {
            cleanup();
            throw;
        }
        cleanup();
        PD_CK(cudaMemcpyAsync(sweeps, &done, sizeof(int), cudaMemcpyHostToDevice, st));
        return;
    }
    static int per_sm[2] = {0, 0};
    int& ps = per_sm[sizeof(T) == 8 ? 1 : 0];
    if (!ps) PD_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, k_jacobi_coop<T>, threads, 0));
    int dev = 0, sms = 0;
    PD_CK(cudaGetDevice(&dev));
    PD_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    int need = (npairs * 32 + threads - 1) / threads;
    int blocks = std::max(1, std::min(need, ps * sm_share(sms)));
    PD_CK(cudaMemsetAsync(bar, 0, 3 * sizeof(unsigned), st));
    void* args[] = {(void*)&secs, (void*)&pair_sec, (void*)&npairs, (void*)&maxnpad, (void*)&max_sweeps,
                    (void*)&W, (void*)&V, (void*)&tol, (void*)&fl, (void*)&rot, (void*)&sweeps, (void*)&bar,
                    (void*)&err};
    PD_CK(cudaLaunchCooperativeKernel((void*)k_jacobi_coop<T>, blocks, threads, args, 0, st));
    PD_LAUNCHED();
}
template void launch_jacobi<double>(const SvdSec*, int, const int*, int, int, int, double*, double*, double, double,
                                    double*, int*, int*, unsigned*, unsigned*, cudaStream_t);
template void launch_jacobi<float>(const SvdSec*, int, const int*, int, int, int, float*, float*, float, double,
                                   double*, int*, int*, unsigned*, unsigned*, cudaStream_t);

template <class T>
void launch_svd_norms(const SvdSec* secs, int nsec, int max_n, const T* W, double* sig, cudaStream_t st) {
    if (nsec <= 0 || max_n <= 0) return;
    k_svd_norms<T><<<dim3((max_n + 7) / 8, nsec), 256, 0, st>>>(secs, W, sig);
    PD_LAUNCHED();
}
template void launch_svd_norms<double>(const SvdSec*, int, int, const double*, double*, cudaStream_t);

template <class T>
void launch_svd_finish(const SvdSec* secs, int nsec, int max_n, const T* W, double* sig, int* order, cudaStream_t st) {
    if (nsec <= 0 || max_n <= 0) return;
    launch_svd_norms<T>(secs, nsec, max_n, W, sig, st);
    k_svd_order<<<dim3((max_n + 7) / 8, nsec), 256, 0, st>>>(secs, sig, order);
    PD_LAUNCHED();
}
template void launch_svd_finish<double>(const SvdSec*, int, int, const double*, double*, int*, cudaStream_t);
template void launch_svd_finish<float>(const SvdSec*, int, int, const float*, double*, int*, cudaStream_t);

void launch_truncate(const SvdSec* secs, int nsec, const double* sig, const int* order, int total, int m_max,
                     double rel_cutoff, double degen_tol, int* kept, double* weights, double* scratch_d, int* scratch_i,
                     cudaStream_t st) {
    PD_REQUIRE(nsec <= 256, DMRG_ERR_CAPACITY, "more than 256 charge sectors on one bond");
    if (total <= 0) return;
    double* lam = scratch_d;
    double* lmax = scratch_d + total;
    int* sec = scratch_i;
    int* rank = scratch_i + total;
    k_trunc_flat<<<nsec, 256, 0, st>>>(secs, nsec, sig, order, lam, sec, lmax);
    PD_LAUNCHED();
    k_trunc_rank<<<(total + 7) / 8, 256, 0, st>>>(lam, total, lmax, nsec, rel_cutoff, rank);
    PD_LAUNCHED();
    k_trunc_count<<<1, 1024, 0, st>>>(lam, sec, rank, total, nsec, m_max, degen_tol, kept, weights);
    PD_LAUNCHED();
}

}  // namespace pd
