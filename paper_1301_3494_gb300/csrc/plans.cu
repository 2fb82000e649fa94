// Contraction plans and device building blocks of the two-site DMRG step (Sec. II).
#include <cfloat>
#include <cmath>
#include <cstring>
#include <map>

#include "plans.h"

namespace pd {

thread_local int g_svd_qr = 1;

// ------------------------------------------------------------------------------------------
// Layouts
// ------------------------------------------------------------------------------------------
SiteLayout site_layout(const Sec& bl, const Sec& br, const std::vector<int>& qn) {
    SiteLayout L;
    L.d = (int)qn.size();
    L.index.assign((size_t)bl.n() * L.d, -1);
    long long off = 0;
    for (int i = 0; i < bl.n(); ++i)
        for (int s = 0; s < L.d; ++s) {
            int j = br.find(bl.q[i] + qn[s]);
            if (j < 0) continue;
            L.index[(size_t)i * L.d + s] = (int)L.blk.size();
            L.blk.push_back({i, s, j, off, bl.m[i], br.m[j]});
            off += (long long)bl.m[i] * br.m[j];
        }
    L.size = off;
    return L;
}

PsiLayout psi_layout2(const Sec& bl, const Sec& br, const std::vector<int>& qn1, const std::vector<int>& qn2) {
    PsiLayout P;
    P.d1 = (int)qn1.size();
    P.d2 = (int)qn2.size();
    P.d = P.d1;
    P.index.assign((size_t)bl.n() * P.d1 * P.d2, -1);
    long long off = 0;
    for (int i = 0; i < bl.n(); ++i)
        for (int s1 = 0; s1 < P.d1; ++s1)
            for (int s2 = 0; s2 < P.d2; ++s2) {
                int k = br.find(bl.q[i] + qn1[s1] + qn2[s2]);
                if (k < 0) continue;
                P.index[((size_t)i * P.d1 + s1) * P.d2 + s2] = (int)P.blk.size();
                P.blk.push_back({i, s1, s2, k, off, bl.m[i], br.m[k]});
                off += (long long)bl.m[i] * br.m[k];
            }
    P.size = off;
    return P;
}

PsiLayout psi_layout(const Sec& bl, const Sec& br, const std::vector<int>& qn) { return psi_layout2(bl, br, qn, qn); }

EnvLayout env_layout(const Sec& b, const std::vector<int>& flux, int ld) {
    EnvLayout E;
    E.D = (int)flux.size();
    E.ld = ld;
    E.index.assign((size_t)b.n() * E.D, -1);
    long long row = 0, packed = 0;
    for (int i = 0; i < b.n(); ++i)
        for (int w = 0; w < E.D; ++w) {
            int k = b.find(b.q[i] - flux[w]);
            if (k < 0) continue;
            E.index[(size_t)i * E.D + w] = (int)E.blk.size();
            E.blk.push_back({i, w, k, row, packed, b.m[i], b.m[k]});
            row += b.m[i];
            packed += (long long)b.m[i] * b.m[k];
        }
    E.rows = row;
    E.packed_size = packed;
    return E;
}

TwoSiteMPO two_site_mpo(const SiteMPO& a, const SiteMPO& b) {
    TwoSiteMPO T;
    const int d = a.d;
    T.D0 = a.Dl;
    T.D2 = b.Dr;
    T.d = d;
    T.f0 = a.fl;
    T.f2 = b.fr;
    // nonzero entries of W2 by its left channel; one left channel's entries are summed in a dense
    // scratch indexed [s1][s1'][s2][s2'][w2]
    struct E2 { int s2, s2p, w2; double y; };
    std::vector<std::vector<E2>> second(b.Dl);
    for (int w1 = 0; w1 < b.Dl; ++w1)
        for (int s2 = 0; s2 < d; ++s2)
            for (int s2p = 0; s2p < d; ++s2p)
                for (int w2 = 0; w2 < b.Dr; ++w2) {
                    const double y = b.at(w1, s2, s2p, w2);
                    if (y != 0.0) second[w1].push_back({s2, s2p, w2, y});
                }
    const int n = d * d * d * d * b.Dr;
    std::vector<double> acc(n, 0.0);
    std::vector<char> seen(n, 0);
    std::vector<int> touched;
    for (int w = 0; w < a.Dl; ++w) {
        touched.clear();
        for (int s1 = 0; s1 < d; ++s1)
            for (int s1p = 0; s1p < d; ++s1p)
                for (int w1 = 0; w1 < a.Dr; ++w1) {
                    const double x = a.at(w, s1, s1p, w1);
                    if (x == 0.0) continue;
                    for (const E2& e : second[w1]) {
                        const int i = (((s1 * d + s1p) * d + e.s2) * d + e.s2p) * b.Dr + e.w2;
                        if (!seen[i]) {
                            seen[i] = 1;
                            touched.push_back(i);
                        }
                        acc[i] += x * e.y;
                    }
                }
        std::sort(touched.begin(), touched.end());
        for (const int i : touched) {
            const int w2 = i % b.Dr, s2p = i / b.Dr % d, s2 = i / b.Dr / d % d, s1p = i / b.Dr / d / d % d;
            if (acc[i] != 0.0) T.nz.push_back({w, i / b.Dr / d / d / d, s1p, s2, s2p, w2, acc[i]});
            acc[i] = 0.0;
            seen[i] = 0;
        }
    }
    return T;
}

// ------------------------------------------------------------------------------------------
// Batches and job lists
// ------------------------------------------------------------------------------------------
static std::vector<GTile> tile_list(const std::vector<GProb>& probs, int tm, int tn) {
    std::vector<GTile> tiles;
    tiles.reserve(probs.size());
    for (int p = 0; p < (int)probs.size(); ++p)
        for (int m0 = 0; m0 < probs[p].M; m0 += tm)
            for (int n0 = 0; n0 < probs[p].N; n0 += tn) tiles.push_back({p, m0, n0, 0});
    return tiles;
}

void GemmBatch::upload_tiles(int tm, int tn, cudaStream_t st) {
    if (tile_m == tm && tile_n == tn && dtiles.p) return;
    const std::vector<GTile> tiles = tile_list(probs, tm, tn);
    ntiles = (int)tiles.size();
    if (!dprobs.p) upload(dprobs, probs, st);
    if (!dsegs.p) upload(dsegs, segs, st);
    upload(dtiles, tiles, st);
    tile_m = tm;
    tile_n = tn;
}

void GemmBatch::stage(ListPack& pk, int tm, int tn) {
    if (empty()) return;
    pk.add(dprobs, probs);
    pk.add(dsegs, segs);
    if (!tm) return;
    const std::vector<GTile> tiles = tile_list(probs, tm, tn);
    ntiles = (int)tiles.size();
    pk.add(dtiles, tiles);
    tile_m = tm;
    tile_n = tn;
}

void GemmBatch::stage_f64(ListPack& pk) {
    if (empty()) return;
    f64 = f64_shape(probs, segs);
    stage(pk, f64.tile, f64.tile);
}

// Whether a batch runs emulated.  Its plan is built on the host (one to several ms for the batches of a
// bond) and a run is seven launches and two host waits around the slice products, so it only pays for
// large batches, or for middling ones whose plan is run many times.  Size and that hint (a Davidson's
// matvec, a polish, a kept measurement plan) decide, never the history of a batch: the two arithmetics round
// differently, and one operator must not change between its applications.  Measured, FP64 units against
// a first emulated run / a repeated one:
//   17 of 320 x 320 x 640 (2.2 GFLOP)        2.1 ms,  2.0 / 1.0 ms
//   68 of 80 x 80, 20 x K = 80 (1.4 GFLOP)   1.5 ms,  4.5 / 1.3 ms
//   68 of 150 x 150, 26 x K = 150 (12)       10 ms,   13 / 5.0 ms
//   2000^3 (16)                              13 ms,   4.3 / 1.8 ms
//   34 of 80 x 80 x 80 (0.035)               0.05 ms, 0.5 / 0.2 ms
static bool emulated(const GemmBatch& g) {
    return g_gemm64_emu == 2 || (g_gemm64_emu && g.flops >= (g.repeated ? 1e9 : 6e9));
}

F64Shape GemmBatch::upload_f64(cudaStream_t st) {
    if (!f64.tile) f64 = f64_shape(probs, segs);
    upload_tiles(f64.tile, f64.tile, st);
    return f64;
}

void run_gemm64(GemmBatch& g, const double* A, const double* B, double* C, cudaStream_t st) {
    if (g.empty()) return;
    if (emulated(g) && run_gemm64_emu(g, A, B, C, st)) return;
    const F64Shape shape = g.upload_f64(st);
    void* tok = prof_on() ? prof_start(st) : nullptr;
    launch_gemm_f64(g.dprobs.as<GProb>(), g.dsegs.as<GSeg>(), g.dtiles.as<GTile>(), g.ntiles, shape.tile, shape, A, B, C,
                    st);
    if (tok) prof_stop(tok, st, g_prof_class == PROF_ENV ? PROF_ENV : PROF_F64, g.flops);
}

void run_gemm32(GemmBatch& g, const float* A, const float* B, float* C, cudaStream_t st) {
    if (g.empty()) return;
    for (const auto& p : g.probs)
        PD_REQUIRE(p.sak == 1 && p.sbk == 1 && p.sam % 16 == 0 && p.sbn % 16 == 0, DMRG_ERR_ARG,
                   "FP32 GEMM needs K-major slabs with padded rows");
    for (const auto& x : g.segs)
        PD_REQUIRE(x.a_off % 4 == 0 && x.b_off % 4 == 0, DMRG_ERR_ARG, "FP32 GEMM needs 16-byte aligned operand rows");
    g.upload_tiles(64, 64, st);
    void* tok = prof_on() ? prof_start(st) : nullptr;
    launch_gemm_f32(g.dprobs.as<GProb>(), g.dsegs.as<GSeg>(), g.dtiles.as<GTile>(), g.ntiles, A, B, C, st);
    if (tok) prof_stop(tok, st, PROF_F32, g.flops);
}

template <class Tin>
void run_copy(const CopyList& c, const Tin* src, void* dst, Num out, cudaStream_t st) {
    if (c.jobs.empty()) return;
    const CopyJob* j = c.d.as<CopyJob>();
    const int2* ch = c.dc.as<int2>();
    int n = c.nchunks;
    if (out == Num::F64) launch_copy<Tin, double>(j, ch, n, src, (double*)dst, st);
    else if (out == Num::F32) launch_copy<Tin, float>(j, ch, n, src, (float*)dst, st);
    else launch_copy<Tin, __nv_bfloat16>(j, ch, n, src, (__nv_bfloat16*)dst, st);
}
template void run_copy<double>(const CopyList&, const double*, void*, Num, cudaStream_t);
template void run_copy<float>(const CopyList&, const float*, void*, Num, cudaStream_t);

template <>
void run_mix<double>(const MixList& m, const double* in, void* out, Num t, cudaStream_t st) {
    if (m.jobs.empty()) return;
    PD_REQUIRE(t == Num::F64, DMRG_ERR_ARG, "FP64 mix output must be FP64");
    launch_mix<double, double>(m.dj.as<MixJob>(), m.dc.as<int2>(), m.nchunks, m.dt.as<MixTerm>(), in, (double*)out, st);
}
template <>
void run_mix<float>(const MixList& m, const float* in, void* out, Num t, cudaStream_t st) {
    if (m.jobs.empty()) return;
    if (t == Num::F32)
        launch_mix<float, float>(m.dj.as<MixJob>(), m.dc.as<int2>(), m.nchunks, m.dt.as<MixTerm>(), in, (float*)out, st);
    else
        launch_mix<float, __nv_bfloat16>(m.dj.as<MixJob>(), m.dc.as<int2>(), m.nchunks, m.dt.as<MixTerm>(), in, (__nv_bfloat16*)out, st);
}

// ------------------------------------------------------------------------------------------
// Small helper kernels local to this file
// ------------------------------------------------------------------------------------------
namespace {

__global__ void k_scale_plain(double* x, long long n, double s) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] *= s;
}

// out block (rows x cols, row-major) = in block with column c scaled by v[voff + c].
struct ColScaleJob { long long src, dst, voff; int rows, cols; };
__global__ void k_colscale(const ColScaleJob* jobs, const double* in, const double* v, double* out) {
    const ColScaleJob j = jobs[blockIdx.y];
    long long total = (long long)j.rows * j.cols;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        int c = (int)(e % j.cols);
        out[j.dst + e] = in[j.src + e] * v[j.voff + c];
    }
}

// SVD scatter: write kept singular vectors into packed site-tensor blocks.
struct ScatJob {
    long long dst;       // output block offset
    long long base;      // W or V sector base offset
    long long s_off;     // sector offset into sig/order
    int rows, cols;      // output block shape
    int ld;              // column length of the source matrix (W: p, V: n)
    int off0;            // row offset inside the source column (r0 or c0)
    int fromW;           // 1: source columns in W (divide by sigma), 0: in V
    int left;            // 1: output [a][t] (t = kept index = column), 0: output [t][c]
    int lam_pow;         // multiply by lambda_t (normalised) when 1
    int pad_;
};
template <class T>
__global__ void k_svd_scatter(const ScatJob* jobs, const T* W, const T* V, const double* sig,
                              const int* order, const double* weights, double* out) {
    const ScatJob j = jobs[blockIdx.y];
    const double nrm = sqrt(weights[1]);
    long long total = (long long)j.rows * j.cols;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        int r = (int)(e / j.cols), c = (int)(e % j.cols);
        int t = j.left ? c : r;          // kept index
        int x = j.left ? r : c;          // position inside the source column
        int col = order[j.s_off + t];
        double sg = sig[j.s_off + col];
        double val = j.fromW ? (double)W[j.base + (long long)col * j.ld + j.off0 + x] / sg
                             : (double)V[j.base + (long long)col * j.ld + j.off0 + x];
        if (j.lam_pow) val *= sg / nrm;
        out[j.dst + e] = val;
    }
}

// lam_out[o + t] = sig[s_off + order[s_off + t]] / nrm
struct LamJob { long long s_off, o; int k, pad_; };
__global__ void k_lam_out(const LamJob* jobs, int njobs, const double* sig, const int* order, const double* weights,
                          double* lam) {
    const double nrm = sqrt(weights[1]);
    for (int b = blockIdx.x; b < njobs; b += gridDim.x) {
        LamJob j = jobs[b];
        for (int t = threadIdx.x; t < j.k; t += blockDim.x) lam[j.o + t] = sig[j.s_off + order[j.s_off + t]] / nrm;
    }
}

inline int gridn(long long n, int cap = 2048) {
    long long g = (n + 255) / 256;
    return (int)std::max<long long>(1, std::min<long long>(g, cap));
}

}  // namespace

namespace {
struct RCJob { long long off, voff; int rows, cols, by_col, pad_; };
__global__ void k_rcscale(const RCJob* jobs, const double* in, const double* v, double* out) {
    const RCJob j = jobs[blockIdx.y];
    long long total = (long long)j.rows * j.cols;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        int r = (int)(e / j.cols), c = (int)(e % j.cols);
        out[j.off + e] = in[j.off + e] * v[j.voff + (j.by_col ? c : r)];
    }
}
}  // namespace

void scale_site(const Sec& bl, const Sec& br, const std::vector<int>& qn, const double* in, const double* lam,
                bool right_index, double* out, cudaStream_t st) {
    const SiteLayout S = site_layout(bl, br, qn);
    const Sec& vb = right_index ? br : bl;
    std::vector<long long> voff(vb.n() + 1, 0);
    for (int i = 0; i < vb.n(); ++i) voff[i + 1] = voff[i] + vb.m[i];
    std::vector<RCJob> jobs;
    int mx = 1;
    for (const auto& b : S.blk) {
        jobs.push_back({b.off, voff[right_index ? b.j : b.i], b.rows, b.cols, right_index ? 1 : 0, 0});
        mx = std::max(mx, b.rows * b.cols);
    }
    if (jobs.empty()) return;
    DBuf dj;
    upload(dj, jobs, st);
    k_rcscale<<<dim3(gridn(mx, 256), (unsigned)jobs.size()), 256, 0, st>>>(dj.as<RCJob>(), in, lam, out);
    PD_LAUNCHED();
    PD_CK(cudaStreamSynchronize(st));
}

namespace {
// Symmetric k x k blocks G_j = sum A^T A at off, formed as the lower triangle only (see add_gram): an
// element (r, c), r >= c, is at off + r + c k.
struct NsJob { long long off; int k, pad_; };
__device__ __forceinline__ double gram_at(const double* G, const NsJob& j, int r, int c) {
    return G[j.off + max(r, c) + (long long)min(r, c) * j.k];
}
// T_j = 1.5 I - 0.5 G_j
__global__ void k_ns_prep(const NsJob* jobs, const double* G, double* T) {
    const NsJob j = jobs[blockIdx.y];
    const int total = j.k * j.k;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int c = e / j.k, r = e - c * j.k;
        T[j.off + e] = (r == c ? 1.5 : 0.0) - 0.5 * gram_at(G, j, r, c);
    }
}
// E_j = G_j - I (both triangles), T_j = I - E_j / 2
__global__ void k_ns_start(const NsJob* jobs, const double* G, double* E, double* T) {
    const NsJob j = jobs[blockIdx.y];
    const int total = j.k * j.k;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int c = e / j.k, r = e - c * j.k;
        const double one = r == c ? 1.0 : 0.0, d = gram_at(G, j, r, c) - one;
        E[j.off + e] = d;
        T[j.off + e] = fma(-0.5, d, one);
    }
}
// S_j's upper triangle from its lower one; E_j <- 3/8 I - 5/16 E_j + 35/128 S_j
__global__ void k_ns_quintic(const NsJob* jobs, double* S, double* E) {
    const NsJob j = jobs[blockIdx.y];
    const int total = j.k * j.k;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int c = e / j.k, r = e - c * j.k;
        const double s = gram_at(S, j, r, c);
        if (r < c) S[j.off + e] = s;
        E[j.off + e] = fma(0.2734375, s, fma(-0.3125, E[j.off + e], r == c ? 0.375 : 0.0));
    }
}
// T_j's upper triangle from its lower one
__global__ void k_mirror(const NsJob* jobs, double* T) {
    const NsJob j = jobs[blockIdx.y];
    const int total = j.k * j.k;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int c = e / j.k, r = e - c * j.k;
        if (r < c) T[j.off + e] = T[j.off + c + (long long)r * j.k];
    }
}
// dev[2 x] = max |G - I|, dev[2 x + 1] = sum of (G - I)^2 over CTA x's columns of block s (x = s gridDim.x +
// blockIdx.x).  CTAs share a block: one CTA each took 1.2 ms for the blocks of an m = 2000 bond.
__global__ void __launch_bounds__(128) k_gram_dev(const NsJob* jobs, const double* G, double* dev) {
    const NsJob j = jobs[blockIdx.y];
    long long m = 0;                                           // magnitudes order like their bits
    double f = 0.0;
    for (int c = blockIdx.x; c < j.k; c += gridDim.x)
        for (int r = c + threadIdx.x; r < j.k; r += blockDim.x) {
            const double d = fabs(G[j.off + r + (long long)c * j.k] - (r == c ? 1.0 : 0.0));
            if (d == d) m = max(m, __double_as_longlong(d));   // (NaN is passed over)
            f = fma(r == c ? d : 2.0 * d, d, f);
        }
    for (int o = 16; o > 0; o >>= 1) {
        m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        f += __shfl_xor_sync(0xffffffffu, f, o);
    }
    __shared__ long long sm[4];
    __shared__ double sf[4];
    if ((threadIdx.x & 31) == 0) {
        sm[threadIdx.x >> 5] = m;
        sf[threadIdx.x >> 5] = f;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double* o = dev + 2 * ((long long)blockIdx.y * gridDim.x + blockIdx.x);
        o[0] = __longlong_as_double(max(max(sm[0], sm[1]), max(sm[2], sm[3])));
        o[1] = (sf[0] + sf[1]) + (sf[2] + sf[3]);
    }
}

// Over all blocks, on the host: max |G - I|, and the largest Frobenius norm of a block's G - I.
struct GramDev { double max, fro; };
GramDev gram_deviation(const DBuf& djobs, const std::vector<NsJob>& jobs, const DBuf& G, DBuf& dev, cudaStream_t st) {
    const int n = (int)jobs.size();
    int kmax = 1;
    for (const NsJob& j : jobs) kmax = std::max(kmax, j.k);
    const int ctas = std::min(kmax, 32);
    std::vector<double> h((size_t)2 * n * ctas);
    dev.ensure(h.size() * 8, st);
    k_gram_dev<<<dim3(ctas, (unsigned)n), 128, 0, st>>>(djobs.as<NsJob>(), G.as<double>(), dev.as<double>());
    PD_LAUNCHED();
    PD_CK(cudaMemcpyAsync(h.data(), dev.p, h.size() * 8, cudaMemcpyDeviceToHost, st));
    PD_CK(cudaStreamSynchronize(st));
    GramDev d{0.0, 0.0};
    for (int s = 0; s < n; ++s) {
        double f = 0.0;
        for (int x = 0; x < ctas; ++x) {
            d.max = std::max(d.max, h[2 * ((size_t)s * ctas + x)]);
            f += h[2 * ((size_t)s * ctas + x) + 1];
        }
        // (a sum that overflowed, or NaN, settles nothing)
        d.fro = f <= 1e30 ? std::max(d.fro, std::sqrt(f)) : 1e30;
    }
    return d;
}

// Adds to g the lower triangle of the k x k Gram block at c_off, 64 columns at a time: half the work of
// the square.  Column i of segment s starts at segs[s].a_off + i sam; strides as for GemmBatch::add.
void add_gram(GemmBatch& g, int k, long long c_off, int sam, int sak, const std::vector<GSeg>& segs, int accumulate = 0,
              double alpha = 1.0) {
    for (int j0 = 0; j0 < k; j0 += 64) {
        std::vector<GSeg> sg = segs;
        for (GSeg& x : sg) {
            x.a_off += (long long)j0 * sam;
            x.b_off = x.a_off;
        }
        g.add(k - j0, std::min(64, k - j0), c_off + j0 + (long long)j0 * k, sam, sak, sam, sak, 1, k, sg, accumulate, alpha);
    }
}

// T ~ G^(-1/2), so that X T has orthonormal columns to `goal` where that is in reach.  With E = G - I,
// the series of (1 + E)^(-1/2) cut after
//   - E / 2 (a Newton-Schulz step)               leaves |X'^T X' - I| <= 3/4 |E|^2,
//   3/8 E^2                                      5/8 |E|^3,
//   E^2 (3/8 - 5/16 E + 35/128 E^2)              63/128 |E|^5
// (spectral norms; the Frobenius norm bounds them).  The shortest whose bound meets the goal is the last
// step: the Gram matrix is not formed again to see it.  From an FP32 Jacobi's rotations (1e-6 to 1e-4 an
// element) that is one Gram matrix, one or two triangular products and one product instead of three Gram
// matrices and two products, and one host wait instead of three: FP64 split of the 512-state chain bond
// 20.3 -> 18.5 ms, accurate split of the cylinder's m = 1000 bond 36.3 -> 31.3, four mixed splits at m =
// 2000 40.1 -> 37.4, a 16-site FP64 sweep at m = 64 115 -> 98.
struct NsStep {
    const DBuf& dj;
    const std::vector<NsJob>& jobs;
    DBuf E, S;
    GemmBatch gT, gS, gP;                 // T += 3/8 E E;  S = E E;  T += S P (lower triangles)
    int mx = 1;
    long long size = 0;
    NsStep(const DBuf& dj_, const std::vector<NsJob>& jobs_) : dj(dj_), jobs(jobs_) {
        for (const NsJob& j : jobs) {
            mx = std::max(mx, j.k * j.k);
            size = std::max(size, j.off + (long long)j.k * j.k);
        }
    }
    void products(GemmBatch& g, int accumulate, double alpha) {
        if (!g.probs.empty()) return;
        for (const NsJob& j : jobs) add_gram(g, j.k, j.off, j.k, 1, {GSeg{j.off, j.off, j.k, 0}}, accumulate, alpha);
    }
    // Returns whether this step was the last one needed.
    bool make(const GramDev& d, double goal, const DBuf& G, DBuf& T, cudaStream_t st) {
        const dim3 grid(gridn(mx, 256), (unsigned)jobs.size());
        const double f = d.fro, f2 = f * f;
        const bool square = 0.75 * f2 <= goal, cubic = 0.625 * f * f2 <= goal, quintic = 63.0 / 128.0 * f * f2 * f2 <= goal;
        if (square || !quintic) {
            k_ns_prep<<<grid, 256, 0, st>>>(dj.as<NsJob>(), G.as<double>(), T.as<double>());
            PD_LAUNCHED();
            return square;
        }
        E.ensure(size * 8, st);
        k_ns_start<<<grid, 256, 0, st>>>(dj.as<NsJob>(), G.as<double>(), E.as<double>(), T.as<double>());
        PD_LAUNCHED();
        if (cubic) {
            products(gT, 1, 0.375);
            run_gemm64(gT, E.as<double>(), E.as<double>(), T.as<double>(), st);
        } else {
            products(gS, 0, 1.0);
            products(gP, 1, 1.0);
            S.ensure(size * 8, st);
            run_gemm64(gS, E.as<double>(), E.as<double>(), S.as<double>(), st);
            k_ns_quintic<<<grid, 256, 0, st>>>(dj.as<NsJob>(), S.as<double>(), E.as<double>());
            PD_LAUNCHED();
            run_gemm64(gP, S.as<double>(), E.as<double>(), T.as<double>(), st);
        }
        k_mirror<<<grid, 256, 0, st>>>(dj.as<NsJob>(), T.as<double>());
        PD_LAUNCHED();
        return true;
    }
};
}  // namespace

void orthonormalize_factor(const Sec& bl, const Sec& br, const std::vector<int>& qn, double* X, bool left,
                           cudaStream_t st) {
    const SiteLayout S = site_layout(bl, br, qn);
    const Sec& mid = left ? br : bl;            // the bond carrying the kept index
    std::vector<long long> goff(mid.n() + 1, 0);
    for (int i = 0; i < mid.n(); ++i) goff[i + 1] = goff[i] + (long long)mid.m[i] * mid.m[i];
    DBuf G, T, out, dev, dj;
    G.ensure(std::max<long long>(1, goff.back()) * 8, st);
    T.ensure(std::max<long long>(1, goff.back()) * 8, st);
    out.ensure(std::max<long long>(1, S.size) * 8, st);
    std::vector<NsJob> jobs;
    for (int j = 0; j < mid.n(); ++j) jobs.push_back({goff[j], mid.m[j], 0});
    upload(dj, jobs, st);
    GemmBatch gA;
    for (const auto& b : S.blk) {
        if (left) {
            int k = b.cols;   // A'[a][t] = sum_u A[a][u] T[u][t]:  C(m = t, n = a)
            gA.add(k, b.rows, b.off, 1, k, k, 1, 1, k, {GSeg{goff[b.j], b.off, k, 0}});
        } else {
            int k = b.rows;   // B'[t][c] = sum_u T[t][u] B[u][c]:  C(m = c, n = t)
            gA.add(b.cols, k, b.off, 1, b.cols, k, 1, 1, b.cols, {GSeg{b.off, goff[b.i], k, 0}});
        }
    }
    // G_j = sum over the blocks of sector j of A^T A (left: all blocks share k_j columns, one problem)
    // or B B^T (right: the blocks' row strides differ, so the n-th block of every sector goes into the
    // n-th, accumulating launch)
    std::vector<GemmBatch> gG;
    if (left) {
        gG.emplace_back();
        std::vector<std::vector<GSeg>> segs(mid.n());
        for (const auto& b : S.blk) segs[b.j].push_back({b.off, b.off, b.rows, 0});
        for (int j = 0; j < mid.n(); ++j) add_gram(gG[0], mid.m[j], goff[j], 1, mid.m[j], segs[j]);
    } else {
        std::vector<int> nth(mid.n(), 0);
        for (const auto& b : S.blk) {
            const int t = nth[b.i]++;
            if ((int)gG.size() <= t) gG.emplace_back();
            add_gram(gG[t], b.rows, goff[b.i], b.cols, 1, {GSeg{b.off, b.off, b.cols, 0}}, t > 0);
        }
    }
    NsStep ns(dj, jobs);
    for (int iter = 0; iter < 6; ++iter) {
        PD_CK(cudaMemsetAsync(G.p, 0, std::max<long long>(1, goff.back()) * 8, st));
        for (auto& g1 : gG) run_gemm64(g1, X, X, G.as<double>(), st);
        const GramDev d = gram_deviation(dj, jobs, G, dev, st);
        const double worst = d.max;
        PD_REQUIRE(std::isfinite(worst) && worst < 0.9, DMRG_ERR_NUMERIC,
                   "kept singular vectors too far from orthonormal for the FP64 re-orthonormalisation (|I - X^T X| = " +
                       std::to_string(worst) + " at iteration " + std::to_string(iter) + ")");
        if (worst < 1e-13 || iter == 5) break;
        // X <- X T (left) or T X (right)
        const bool last = ns.make(d, 1e-13, G, T, st);
        if (left) run_gemm64(gA, T.as<double>(), X, out.as<double>(), st);
        else run_gemm64(gA, X, T.as<double>(), out.as<double>(), st);
        PD_CK(cudaMemcpyAsync(X, out.p, S.size * 8, cudaMemcpyDeviceToDevice, st));
        if (last) break;
    }
    PD_CK(cudaStreamSynchronize(st));
}

void convert_flat(const void* src, Num in, void* dst, Num out, long long n, cudaStream_t st) {
    PD_REQUIRE(in != out && (in == Num::F64 || in == Num::F32), DMRG_ERR_ARG, "convert_flat: unsupported types");
    if (in == Num::F64) {
        const double* s = static_cast<const double*>(src);
        if (out == Num::F32) launch_convert(s, static_cast<float*>(dst), n, st);
        else launch_convert(s, static_cast<__nv_bfloat16*>(dst), n, st);
    } else {
        const float* s = static_cast<const float*>(src);
        if (out == Num::F64) launch_convert(s, static_cast<double*>(dst), n, st);
        else launch_convert(s, static_cast<__nv_bfloat16*>(dst), n, st);
    }
}

bool orthonormalize_square(const std::vector<SvdSec>& ss, double* V, cudaStream_t st, int steps) {
    std::vector<NsJob> jobs;
    GemmBatch gG, gX;
    long long tot = 0, first = 0, sum = 0;
    for (const auto& x : ss) {
        if (x.n <= 0) continue;
        const int n = x.n;
        if (jobs.empty()) first = x.v_off;
        jobs.push_back({x.v_off, n, 0});
        sum += (long long)n * n;
        // G = V^T V:  G(i, j) = sum_k V(k, i) V(k, j), V column-major (V(r, c) = V[off + r + c n])
        add_gram(gG, n, x.v_off, n, 1, {GSeg{x.v_off, x.v_off, n, 0}});
        // V' = V T:   V'(r, c) = sum_u V(r, u) T(u, c), T symmetric
        gX.add(n, n, x.v_off, 1, n, n, 1, 1, n, {GSeg{x.v_off, x.v_off, n, 0}});
        tot = std::max(tot, x.v_off + (long long)n * n);
    }
    if (jobs.empty()) return true;
    PD_REQUIRE(sum == tot - first, DMRG_ERR_STATE, "sector matrices are not contiguous");
    DBuf G, T, out, dev, dj;
    G.ensure(tot * 8, st);
    T.ensure(tot * 8, st);
    out.ensure(tot * 8, st);
    upload(dj, jobs, st);
    NsStep ns(dj, jobs);
    for (int iter = 0; iter < steps; ++iter) {
        run_gemm64(gG, V, V, G.as<double>(), st);
        const GramDev d = gram_deviation(dj, jobs, G, dev, st);
        const double worst = d.max;
        PD_REQUIRE(std::isfinite(worst) && worst < 0.5, DMRG_ERR_NUMERIC,
                   "FP32 Jacobi rotations too far from orthogonal for the FP64 polish (|V^T V - I| = " +
                       std::to_string(worst) + " at iteration " + std::to_string(iter) + ")");
        if (worst < 1e-14) return true;
        const bool last = ns.make(d, 1e-14, G, T, st);
        run_gemm64(gX, V, T.as<double>(), out.as<double>(), st);
        // the matrices follow each other without gaps
        PD_CK(cudaMemcpyAsync(V + first, out.as<double>() + first, (size_t)(tot - first) * 8, cudaMemcpyDeviceToDevice, st));
        if (last) return true;
    }
    return false;
}

void scale_vec(double* x, long long n, double s, cudaStream_t st) {
    if (n <= 0) return;
    k_scale_plain<<<gridn(n), 256, 0, st>>>(x, n, s);
    PD_LAUNCHED();
}

double dot_host(const double* x, const double* y, long long n, cudaStream_t st) {
    DBuf part, out;
    int nch = 64;
    part.ensure(sizeof(double) * nch, st);
    out.ensure(sizeof(double), st);
    launch_dots(x, 0, 1, y, n, part.as<double>(), nch, out.as<double>(), st);
    double h = 0.0;
    PD_CK(cudaMemcpyAsync(&h, out.p, sizeof(double), cudaMemcpyDeviceToHost, st));
    PD_CK(cudaStreamSynchronize(st));
    return h;
}

// ------------------------------------------------------------------------------------------
// Projected Hamiltonian plan: out = L x W1 x W2 x R applied to psi
// ------------------------------------------------------------------------------------------
std::unique_ptr<HeffPlan> make_heff_plan(const Sec& bl, const Sec& br, const std::vector<int>& qn,
                                         const TwoSiteMPO& w12, const EnvLayout& L, const EnvLayout& R,
                                         int prec, cudaStream_t st) {
    auto P = std::make_unique<HeffPlan>();
    const int d = (int)qn.size();
    P->prec = prec;
    P->psi = psi_layout(bl, br, qn);
    P->L = &L;
    P->R = &R;
    P->ld_psi = pad_ld(bl.maxm(), prec);
    P->ld_y = pad_ld(br.maxm(), prec);
    // FP64 plans read any stride (also the tensor-core layout of FP64-accurate mixed-mode
    // environments); the tensor-core plans need the 64-padded operand layout
    PD_REQUIRE(prec == DMRG_FP64 ? (L.ld >= bl.maxm() && R.ld >= br.maxm())
                                 : (L.ld == pad_ld(bl.maxm(), prec) && R.ld == pad_ld(br.maxm(), prec)),
               DMRG_ERR_STATE, "environment slab stride does not match the bond");
    const auto& pb = P->psi.blk;
    const int nb = (int)pb.size();

    // pack x (canonical [a][c]) into the transposed operand slab psiT ([c][a] rows)
    std::vector<long long> prow(nb);
    long long row = 0;
    for (int b = 0; b < nb; ++b) {
        prow[b] = row;
        CopyJob j{};
        j.src = pb[b].off; j.dst = row * P->ld_psi;
        j.rows = pb[b].cols; j.cols = pb[b].rows;
        j.srs = 1; j.scs = pb[b].cols; j.drs = P->ld_psi; j.dcs = 1;
        j.zero_to = kpad(pb[b].rows, prec); j.scale = 1.0;
        P->pack.add(j);
        row += pb[b].cols;
    }
    P->psiT_rows = row;

    // nonzero two-site entries by (s1, s2), ordered by w'' (and as listed within it)
    std::vector<std::vector<int>> by_out((size_t)d * d);
    for (int e = 0; e < (int)w12.nz.size(); ++e) by_out[(size_t)w12.nz[e].s1 * d + w12.nz[e].s2].push_back(e);
    for (auto& v : by_out)
        std::stable_sort(v.begin(), v.end(), [&](int x, int y) { return w12.nz[x].w2 < w12.nz[y].w2; });
    // which (w, s1', s2') combinations feed anything
    std::vector<char> used((size_t)w12.D0 * d * d, 0);
    for (const auto& e : w12.nz) used[((size_t)e.w * d + e.s1p) * d + e.s2p] = 1;

    // L stage: X[w, b] = L_w psi_b, block [a_bra][c].  X blocks that feed exactly one Y block,
    // and that Y block has no other term, are written by the GEMM epilogue straight into the Y
    // operand slab (coefficient as alpha); only the rest goes through X and the mixing kernel.
    struct XB { int rows, cols, lb, b; long long off; int fan; };
    std::vector<XB> xs;
    std::vector<int> xidx((size_t)w12.D0 * nb, -1);   // (w, b) -> X block
    std::vector<int> raised((size_t)w12.D0 * bl.n()), lowered((size_t)w12.D0 * bl.n());
    for (int w = 0; w < w12.D0; ++w)                  // left sector reached from i by channel w, and back
        for (int i = 0; i < bl.n(); ++i) {
            raised[(size_t)w * bl.n() + i] = bl.find(bl.q[i] + w12.f0[w]);
            lowered[(size_t)w * bl.n() + i] = bl.find(bl.q[i] - w12.f0[w]);
        }
    for (int b = 0; b < nb; ++b) {
        const auto& B = pb[b];
        for (int w = 0; w < w12.D0; ++w) {
            if (!used[((size_t)w * d + B.s1) * d + B.s2]) continue;
            const int iab = raised[(size_t)w * bl.n() + B.i];
            if (iab < 0) continue;
            const int lb = L.at(iab, w);
            if (lb < 0) continue;
            xidx[(size_t)w * nb + b] = (int)xs.size();
            xs.push_back({bl.m[iab], B.cols, lb, b, -1, 0});
        }
    }
    // MPO mix: Y[w2, o] = sum coef X[w, b]   (o = output block (iab, s1, s2))
    struct YB { int o, rb, t0, nt; long long row; };
    std::vector<YB> ys;
    std::vector<std::pair<int, double>> yt;           // terms of the Y blocks: (X block, coefficient)
    long long yrow = 0;
    for (int o = 0; o < nb; ++o) {
        const auto& O = pb[o];
        int last = -1;
        for (const int ei : by_out[(size_t)O.s1 * d + O.s2]) {
            const auto& e = w12.nz[ei];
            const int i = lowered[(size_t)e.w * bl.n() + O.i];
            const int b = i < 0 ? -1 : P->psi.at(i, e.s1p, e.s2p);
            const int xi = b < 0 ? -1 : xidx[(size_t)e.w * nb + b];
            if (xi < 0) continue;
            const int rb = R.at(O.k, e.w2);
            if (rb < 0) continue;
            PD_REQUIRE(R.blk[rb].k == pb[b].k, DMRG_ERR_QN, "MPO flux rule violated in the two-site operator");
            if (e.w2 != last) {
                ys.push_back({o, rb, (int)yt.size(), 0, yrow});
                yrow += xs[xi].rows;
                last = e.w2;
            }
            yt.push_back({xi, e.v});
            ys.back().nt++;
            xs[xi].fan++;
        }
    }
    P->y_rows = yrow;
    // direct targets
    std::vector<int> direct(xs.size(), -1);
    for (int y = 0; y < (int)ys.size(); ++y)
        if (ys[y].nt == 1 && xs[yt[ys[y].t0].first].fan == 1) direct[yt[ys[y].t0].first] = y;
    long long xoff = 0;
    for (size_t xi = 0; xi < xs.size(); ++xi) {
        XB& x = xs[xi];
        const auto& B = pb[x.b];
        const GSeg sg{prow[x.b] * P->ld_psi, L.blk[x.lb].row * L.ld, B.rows, 0};
        if (direct[xi] >= 0) {
            const YB& y = ys[direct[xi]];
            P->ldirect.add(x.cols, x.rows, y.row * P->ld_y, P->ld_psi, 1, L.ld, 1, 1, P->ld_y, &sg, 1, 0, yt[y.t0].second);
        } else {
            x.off = xoff;
            P->lstage.add(x.cols, x.rows, xoff, P->ld_psi, 1, L.ld, 1, 1, x.cols, &sg, 1, 0, 1.0);
            xoff += (long long)x.rows * x.cols;
        }
    }
    P->x_size = xoff;
    // mixing jobs for the remaining Y blocks, R-stage segments for all of them
    std::vector<GSeg> rs;
    for (size_t y = 0; y < ys.size();) {
        const int o = ys[y].o;
        rs.clear();
        for (; y < ys.size() && ys[y].o == o; ++y) {
            const YB& Y = ys[y];
            const int x0i = yt[Y.t0].first;
            const XB& x0 = xs[x0i];
            P->mix.flops += 2.0 * x0.rows * x0.cols * (double)Y.nt;
            if (direct[x0i] != (int)y) {
                MixJob mj{};
                mj.dst = Y.row * P->ld_y;
                mj.rows = x0.rows;
                mj.cols = x0.cols;
                mj.ldo = P->ld_y;
                mj.zero_to = kpad(x0.cols, prec);
                mj.t0 = (int)P->mix.terms.size();
                mj.nt = Y.nt;
                for (int t = Y.t0; t < Y.t0 + Y.nt; ++t)
                    P->mix.terms.push_back({xs[yt[t].first].off, xs[yt[t].first].cols, 0, yt[t].second});
                P->mix.jobs.push_back(mj);
            }
            rs.push_back({R.blk[Y.rb].row * R.ld, Y.row * P->ld_y, x0.cols, 0});
        }
        const auto& O = pb[o];
        P->rstage.add(O.cols, O.rows, O.off, R.ld, 1, P->ld_y, 1, 1, O.cols, rs);
    }

    // diagonal
    for (int b = 0; b < nb; ++b) {
        const auto& B = pb[b];
        DiagJob j{};
        j.off = B.off; j.rows = B.rows; j.cols = B.cols; j.t0 = (int)P->dterms.size(); j.nt = 0;
        for (const auto& e : w12.nz) {
            if (e.s1 != B.s1 || e.s1p != B.s1 || e.s2 != B.s2 || e.s2p != B.s2) continue;
            if (w12.f0[e.w] != 0 || w12.f2[e.w2] != 0) continue;
            int lb = L.at(B.i, e.w), rb = R.at(B.k, e.w2);
            if (lb < 0 || rb < 0) continue;
            P->dterms.push_back({L.blk[lb].row * L.ld, R.blk[rb].row * R.ld, e.v});
            ++j.nt;
        }
        P->djobs.push_back(j);
    }

    P->flops = P->lstage.flops + P->ldirect.flops + P->rstage.flops + P->mix.flops;
    // every static list in one upload
    const Num t = mv_num(prec);
    {
        ListPack pk;
        P->pack.stage(pk);
        P->mix.stage(pk);
        pk.add(P->ddj, P->djobs);
        pk.add(P->ddt, P->dterms);
        std::vector<long long> el;
        for (const auto& j : P->djobs) el.push_back((long long)j.rows * j.cols);
        const std::vector<int2> c = make_chunks(el);
        P->diag_chunks = (int)c.size();
        pk.add(P->ddc, c);
        auto stage = [&](GemmBatch& g, Num cnum) {
            g.repeated = true;
            if (prec == DMRG_FP64) g.stage_f64(pk);
            else if (prec == PREC_F32) g.stage(pk, 64, 64);
            else {
                const int bn = g.empty() ? 0 : tc_width(g, t, cnum, true);
                g.stage(pk, bn ? TC_TILE_M : 0, bn);
            }
        };
        stage(P->lstage, Num::F32);
        stage(P->ldirect, t);
        stage(P->rstage, Num::F64);
        pk.upload(P->lists, st);
    }
    P->psiT.ensure(std::max<long long>(1, P->psiT_rows) * P->ld_psi * num_size(t), st);
    P->Y.ensure(std::max<long long>(1, P->y_rows) * P->ld_y * num_size(t), st);
    // directly written Y blocks rely on zero padding columns: clear the slab once
    PD_CK(cudaMemsetAsync(P->Y.p, 0, std::max<long long>(1, P->y_rows) * P->ld_y * num_size(t), st));
    P->X.ensure(std::max<long long>(1, P->x_size) * (prec == DMRG_FP64 ? 8 : 4), st);
    PD_REQUIRE(P->psi.size < (1LL << 31), DMRG_ERR_CAPACITY, "two-site vector too long for one copy job");
    return P;
}

static const void* env_operand(const EnvSlab& e, int prec) {
    if (prec == DMRG_BF16) {
        PD_REQUIRE(e.op_valid, DMRG_ERR_STATE, "bf16 operand copy of an environment is stale");
        return e.op.p;
    }
    if ((prec == DMRG_TF32 || prec == PREC_F32) && e.num == Num::F64) {
        PD_REQUIRE(e.op32_valid, DMRG_ERR_STATE, "FP32 operand copy of an environment is stale");
        return e.op32.p;
    }
    return e.buf.p;
}

void heff_apply(HeffPlan& P, const EnvSlab& L, const EnvSlab& R, const double* x, double* y,
                unsigned* err, cudaStream_t st) {
    g_prof_class = PROF_MV;
    const int prec = P.prec;
    const Num t = mv_num(prec);
    run_copy<double>(P.pack, x, P.psiT.p, t, st);
    PD_CK(cudaMemsetAsync(y, 0, sizeof(double) * std::max<long long>(P.psi.size, 1), st));
    if (prec == DMRG_FP64) {
        run_gemm64(P.lstage, P.psiT.as<double>(), L.buf.as<double>(), P.X.as<double>(), st);
        run_gemm64(P.ldirect, P.psiT.as<double>(), L.buf.as<double>(), P.Y.as<double>(), st);
        run_mix<double>(P.mix, P.X.as<double>(), P.Y.p, Num::F64, st);
        run_gemm64(P.rstage, R.buf.as<double>(), P.Y.as<double>(), y, st);
    } else if (prec == PREC_F32) {
        // accurate refinement matvec: FP32 everywhere, FP64 output
        DBuf y32;
        y32.ensure(std::max<long long>(1, P.psi.size) * 4, st);
        PD_CK(cudaMemsetAsync(y32.p, 0, std::max<long long>(1, P.psi.size) * 4, st));
        const float* Lf = static_cast<const float*>(env_operand(L, PREC_F32));
        const float* Rf = static_cast<const float*>(env_operand(R, PREC_F32));
        run_gemm32(P.lstage, P.psiT.as<float>(), Lf, P.X.as<float>(), st);
        run_gemm32(P.ldirect, P.psiT.as<float>(), Lf, P.Y.as<float>(), st);
        run_mix<float>(P.mix, P.X.as<float>(), P.Y.p, Num::F32, st);
        run_gemm32(P.rstage, Rf, P.Y.as<float>(), y32.as<float>(), st);
        convert_flat(y32.p, Num::F32, y, Num::F64, P.psi.size, st);
    } else {
        run_gemm_tc(P.lstage, t, P.psiT.p, P.psiT_rows, P.ld_psi, env_operand(L, prec), L.lay.rows, L.lay.ld,
                    P.X.p, Num::F32, err, st);
        run_gemm_tc(P.ldirect, t, P.psiT.p, P.psiT_rows, P.ld_psi, env_operand(L, prec), L.lay.rows, L.lay.ld,
                    P.Y.p, t, err, st);
        run_mix<float>(P.mix, P.X.as<float>(), P.Y.p, t, st);
        run_gemm_tc(P.rstage, t, env_operand(R, prec), R.lay.rows, R.lay.ld, P.Y.p, P.y_rows, P.ld_y, y, Num::F64,
                    err, st);
    }
}

void heff_diag(HeffPlan& P, const EnvSlab& L, const EnvSlab& R, double* out, cudaStream_t st) {
    if (P.djobs.empty()) return;
    if (L.num == Num::F64)
        launch_diag<double>(P.ddj.as<DiagJob>(), P.ddc.as<int2>(), P.diag_chunks, P.ddt.as<DiagTerm>(),
                            L.buf.as<double>(), L.lay.ld, R.buf.as<double>(), R.lay.ld, out, st);
    else
        launch_diag<float>(P.ddj.as<DiagJob>(), P.ddc.as<int2>(), P.diag_chunks, P.ddt.as<DiagTerm>(),
                           L.buf.as<float>(), L.lay.ld, R.buf.as<float>(), R.lay.ld, out, st);
}

// ------------------------------------------------------------------------------------------
// Environment slabs
// ------------------------------------------------------------------------------------------
void env_alloc(EnvSlab& e, const Sec& b, const std::vector<int>& flux, int prec, cudaStream_t st) {
    e.lay = env_layout(b, flux, pad_ld(b.maxm(), prec));
    e.num = env_num(prec);
    size_t bytes = (size_t)std::max<long long>(1, e.lay.rows) * e.lay.ld * num_size(e.num);
    e.buf.ensure(bytes, st);
    PD_CK(cudaMemsetAsync(e.buf.p, 0, bytes, st));
    e.op_valid = false;
    e.op32_valid = false;
    e.valid = true;
}

void env_make_operand(EnvSlab& e, int prec, cudaStream_t st) {
    const bool bf = prec == DMRG_BF16, f32 = (prec == DMRG_TF32 || prec == PREC_F32) && e.num == Num::F64;
    if ((!bf && !f32) || (bf && e.op_valid) || (f32 && e.op32_valid)) return;
    // the whole slab (padding included, zeros stay zeros)
    const long long n = std::max<long long>(1, e.lay.rows) * e.lay.ld;
    DBuf& dst = bf ? e.op : e.op32;
    dst.ensure(n * (bf ? 2 : 4), st);
    convert_flat(e.buf.p, e.num, dst.p, bf ? Num::BF16 : Num::F32, n, st);
    (bf ? e.op_valid : e.op32_valid) = true;
}

// Copies of the packed blocks into the slab (lists in one upload).
static CopyList packed_copies(const EnvLayout& lay, DBuf& lists, cudaStream_t st) {
    CopyList c;
    for (const auto& b : lay.blk) {
        CopyJob j{};
        j.src = b.packed; j.dst = b.row * lay.ld; j.rows = b.rows; j.cols = b.cols;
        j.srs = b.cols; j.scs = 1; j.drs = lay.ld; j.dcs = 1; j.zero_to = 0; j.scale = 1.0;
        c.add(j);
    }
    ListPack pk;
    c.stage(pk);
    pk.upload(lists, st);
    return c;
}

void env_from_packed(EnvSlab& e, const double* packed, cudaStream_t st) {
    DBuf lists;
    const CopyList c = packed_copies(e.lay, lists, st);
    run_copy<double>(c, packed, e.buf.p, e.num, st);
    e.op_valid = false;
    e.op32_valid = false;
    e.valid = true;
}

void env_operand_from_packed(EnvSlab& e, const Sec& b, const std::vector<int>& flux, int prec, const double* packed,
                             cudaStream_t st) {
    if (prec != DMRG_BF16) {
        env_alloc(e, b, flux, prec, st);
        env_from_packed(e, packed, st);
        return;
    }
    e.lay = env_layout(b, flux, pad_ld(b.maxm(), prec));
    e.num = env_num(prec);
    const size_t bytes = (size_t)std::max<long long>(1, e.lay.rows) * e.lay.ld * 2;
    e.op.ensure(bytes, st);
    PD_CK(cudaMemsetAsync(e.op.p, 0, bytes, st));
    DBuf lists;
    const CopyList c = packed_copies(e.lay, lists, st);
    run_copy<double>(c, packed, e.op.p, Num::BF16, st);
    e.op_valid = true;
}

void env_to_packed(const EnvSlab& e, double* packed, cudaStream_t st) {
    CopyList c;
    for (const auto& b : e.lay.blk) {
        CopyJob j{};
        j.src = b.row * e.lay.ld; j.dst = b.packed; j.rows = b.rows; j.cols = b.cols;
        j.srs = e.lay.ld; j.scs = 1; j.drs = b.cols; j.dcs = 1; j.zero_to = 0; j.scale = 1.0;
        c.add(j);
    }
    ListPack pk;
    DBuf lists;
    c.stage(pk);
    pk.upload(lists, st);
    if (e.num == Num::F64) run_copy<double>(c, e.buf.as<double>(), packed, Num::F64, st);
    else run_copy<float>(c, e.buf.as<float>(), packed, Num::F64, st);
    PD_CK(cudaStreamSynchronize(st));   // the job list is freed on return
}

void env_boundary(EnvSlab& e, const Sec& b, const std::vector<int>& flux, int prec, cudaStream_t st) {
    env_alloc(e, b, flux, prec, st);
    PD_REQUIRE(e.lay.blk.size() == 1 && e.lay.blk[0].rows == 1 && e.lay.blk[0].cols == 1, DMRG_ERR_QN,
               "boundary environment is not a single 1x1 block");
    if (e.num == Num::F64) {
        double one = 1.0;
        PD_CK(cudaMemcpyAsync(e.buf.p, &one, 8, cudaMemcpyHostToDevice, st));
    } else {
        float one = 1.0f;
        PD_CK(cudaMemcpyAsync(e.buf.p, &one, 4, cudaMemcpyHostToDevice, st));
    }
    PD_CK(cudaStreamSynchronize(st));
    e.op_valid = false;
    e.op32_valid = false;
}

// ------------------------------------------------------------------------------------------
// Environment updates (Sec. II operator transformation)
// ------------------------------------------------------------------------------------------
// Environment updates compound their rounding errors site after site, so they run at FP32
// accuracy or better in every mode: FP64 GEMMs in FP64 mode and, with FP64-accurate environments,
// in the mixed modes (PREC_ENV64, on the tensor-core operand layout); FP32 SIMT GEMMs otherwise.
static void run_env_gemm(GemmBatch& g, int prec, const void* A, long long arows, int lda, const void* B,
                         long long brows, int ldb, void* C, unsigned* err, cudaStream_t st) {
    (void)arows; (void)lda; (void)brows; (void)ldb; (void)err;
    if (g.empty()) return;
    if (env_num(prec) == Num::F64) run_gemm64(g, (const double*)A, (const double*)B, (double*)C, st);
    else run_gemm32(g, (const float*)A, (const float*)B, (float*)C, st);
}

namespace {
// Environment-update GEMMs are tallied as such; the calling thread's class is restored on return.
struct EnvProfClass {
    int saved = g_prof_class;
    EnvProfClass() { g_prof_class = PROF_ENV; }
    ~EnvProfClass() { g_prof_class = saved; }
};
}  // namespace

// Every list of an environment update in one upload (`lists` owns them).
static void stage_env_lists(CopyList& pk, MixList& mx, GemmBatch& g1, GemmBatch& g3, int prec, DBuf& lists,
                            cudaStream_t st) {
    ListPack all;
    pk.stage(all);
    mx.stage(all);
    for (GemmBatch* g : {&g1, &g3})
        if (env_num(prec) == Num::F64) g->stage_f64(all);
        else g->stage(all, 64, 64);
    all.upload(lists, st);
}

void env_update_left(const Sec& ba, const Sec& bb, const std::vector<int>& qn, const SiteMPO& W,
                     const EnvSlab& Lin, const double* A, EnvSlab& Lout, int prec, unsigned* err, cudaStream_t st) {
    EnvProfClass prof_class;
    const int d = (int)qn.size();
    const SiteLayout S = site_layout(ba, bb, qn);
    const EnvLayout& Li = Lin.lay;
    const Num tn = env_num(prec);
    const int ldS = pad_ld(ba.maxm(), prec);
    // A^T slab: block (ia, s) rows b, cols a
    DBuf lists;
    CopyList pk;
    std::vector<long long> srow(S.blk.size());
    long long row = 0;
    for (size_t b = 0; b < S.blk.size(); ++b) {
        const auto& B = S.blk[b];
        srow[b] = row;
        CopyJob j{};
        j.src = B.off; j.dst = row * ldS; j.rows = B.cols; j.cols = B.rows;
        j.srs = 1; j.scs = B.cols; j.drs = ldS; j.dcs = 1; j.zero_to = kpad(B.rows, prec); j.scale = 1.0;
        pk.add(j);
        row += B.cols;
    }
    const long long srows = row;
    // nonzero entries (w, s') of W by (w', s), and which (w, s') feed anything
    struct WE { int w, sp; double c; };
    std::vector<std::vector<WE>> went((size_t)W.Dr * d);
    std::vector<char> usedws((size_t)W.Dl * d, 0);
    for (int w = 0; w < W.Dl; ++w)
        for (int s = 0; s < d; ++s)
            for (int sp = 0; sp < d; ++sp)
                for (int wp = 0; wp < W.Dr; ++wp) {
                    const double c = W.at(w, s, sp, wp);
                    if (c == 0.0) continue;
                    usedws[(size_t)w * d + sp] = 1;
                    went[(size_t)wp * d + s].push_back({w, sp, c});
                }
    // stage 1: T1(iab, w, s') [b][a_bra] = L_w A_s'
    struct TB { long long off; int rows, cols; };   // rows = b, cols = a_bra
    std::vector<TB> t1;
    std::vector<int> t1idx((size_t)ba.n() * W.Dl * d, -1);
    GemmBatch g1;
    long long toff = 0;
    for (const auto& lb : Li.blk) {
        for (int sp = 0; sp < d; ++sp) {
            if (!usedws[(size_t)lb.w * d + sp]) continue;
            int ab = S.at(lb.k, sp);
            if (ab < 0) continue;
            const auto& AB = S.blk[ab];
            t1idx[((size_t)lb.i * W.Dl + lb.w) * d + sp] = (int)t1.size();
            t1.push_back({toff, AB.cols, lb.rows});
            const GSeg sg{lb.row * Li.ld, srow[ab] * ldS, lb.cols, 0};
            g1.add(lb.rows, AB.cols, toff, Li.ld, 1, ldS, 1, 1, lb.rows, &sg, 1, 0, 1.0);
            toff += (long long)AB.cols * lb.rows;
        }
    }
    // stage 2: T2(w', s, iab) [b][a_bra] = sum W[w,s,s',w'] T1(iab, w, s')
    const EnvLayout& Lo = Lout.lay;
    const int ldT = pad_ld(ba.maxm(), prec);
    MixList mx;
    std::vector<long long> t2row((size_t)W.Dr * d * ba.n(), -1);
    long long trow = 0;
    for (int wp = 0; wp < W.Dr; ++wp)
        for (int s = 0; s < d; ++s) {
            const std::vector<WE>& we = went[(size_t)wp * d + s];
            if (we.empty()) continue;
            for (int iab = 0; iab < ba.n(); ++iab) {
                if (S.at(iab, s) < 0) continue;
                const int ibb = bb.find(ba.q[iab] + qn[s]);
                if (ibb < 0 || Lo.at(ibb, wp) < 0) continue;
                const int first = (int)mx.terms.size();
                const TB* x0 = nullptr;
                for (const WE& e : we) {
                    const int ti = t1idx[((size_t)iab * W.Dl + e.w) * d + e.sp];
                    if (ti < 0) continue;
                    x0 = x0 ? x0 : &t1[ti];
                    mx.terms.push_back({t1[ti].off, t1[ti].cols, 0, e.c});
                }
                if (!x0) continue;
                t2row[((size_t)wp * d + s) * ba.n() + iab] = trow;
                MixJob mj{};
                mj.dst = trow * ldT; mj.rows = x0->rows; mj.cols = x0->cols; mj.ldo = ldT;
                mj.zero_to = kpad(x0->cols, prec); mj.t0 = first; mj.nt = (int)mx.terms.size() - first;
                mx.jobs.push_back(mj);
                trow += x0->rows;
            }
        }
    // stage 3: Lout(ibb, w') [b_bra][b] = sum_{s, iab} A_s^T T2(w', s, iab)
    GemmBatch g3;
    std::vector<GSeg> sg;
    for (const auto& ob : Lo.blk) {
        sg.clear();
        for (int s = 0; s < d; ++s) {
            int iab = ba.find(bb.q[ob.i] - qn[s]);
            if (iab < 0) continue;
            int ab = S.at(iab, s);
            if (ab < 0) continue;
            const long long tr = t2row[((size_t)ob.w * d + s) * ba.n() + iab];
            if (tr < 0) continue;
            sg.push_back({tr * ldT, srow[ab] * ldS, ba.m[iab], 0});
        }
        g3.add(ob.cols, ob.rows, ob.row * Lo.ld, ldT, 1, ldS, 1, 1, Lo.ld, sg);
    }
    // execute
    stage_env_lists(pk, mx, g1, g3, prec, lists, st);
    DBuf sl, t1b, t2b;
    sl.ensure(std::max<long long>(1, srows) * ldS * num_size(tn), st);
    t1b.ensure(std::max<long long>(1, toff) * num_size(tn), st);
    t2b.ensure(std::max<long long>(1, trow) * ldT * num_size(tn), st);
    run_copy<double>(pk, A, sl.p, tn, st);
    run_env_gemm(g1, prec, Lin.buf.p, Li.rows, Li.ld, sl.p, srows, ldS, t1b.p, err, st);
    if (tn == Num::F64) run_mix<double>(mx, t1b.as<double>(), t2b.p, tn, st);
    else run_mix<float>(mx, t1b.as<float>(), t2b.p, tn, st);
    run_env_gemm(g3, prec, t2b.p, trow, ldT, sl.p, srows, ldS, Lout.buf.p, err, st);
    Lout.op_valid = false;
    Lout.op32_valid = false;
    PD_CK(cudaStreamSynchronize(st));   // scratch and job lists are released on return
}

void env_update_right(const Sec& ba, const Sec& bc, const std::vector<int>& qn, const SiteMPO& W,
                      const EnvSlab& Rin, const double* Bt, EnvSlab& Rout, int prec, unsigned* err, cudaStream_t st) {
    EnvProfClass prof_class;
    const int d = (int)qn.size();
    const SiteLayout S = site_layout(ba, bc, qn);
    const EnvLayout& Ri = Rin.lay;
    const Num tn = env_num(prec);
    const int ldS = pad_ld(bc.maxm(), prec);
    // B slab: block (ia, s) rows a, cols c (same orientation as the packed block)
    DBuf lists;
    CopyList pk;
    std::vector<long long> srow(S.blk.size());
    long long row = 0;
    for (size_t b = 0; b < S.blk.size(); ++b) {
        const auto& B = S.blk[b];
        srow[b] = row;
        CopyJob j{};
        j.src = B.off; j.dst = row * ldS; j.rows = B.rows; j.cols = B.cols;
        j.srs = B.cols; j.scs = 1; j.drs = ldS; j.dcs = 1; j.zero_to = kpad(B.cols, prec); j.scale = 1.0;
        pk.add(j);
        row += B.rows;
    }
    const long long srows = row;
    // nonzero entries (w', s') of W by (w, s), and which (w', s') feed anything
    struct WE { int wp, sp; double c; };
    std::vector<std::vector<WE>> went((size_t)W.Dl * d);
    std::vector<char> usedws((size_t)W.Dr * d, 0);
    for (int wp = 0; wp < W.Dr; ++wp)
        for (int w = 0; w < W.Dl; ++w)
            for (int s = 0; s < d; ++s)
                for (int sp = 0; sp < d; ++sp) {
                    const double c = W.at(w, s, sp, wp);
                    if (c == 0.0) continue;
                    usedws[(size_t)wp * d + sp] = 1;
                    went[(size_t)w * d + s].push_back({wp, sp, c});
                }
    // stage 1: T1(icb, w', s') [a][c_bra] = R_w' B_s'^T
    struct TB { long long off; int rows, cols; };   // rows = a, cols = c_bra
    std::vector<TB> t1;
    std::vector<int> t1idx((size_t)bc.n() * W.Dr * d, -1);
    GemmBatch g1;
    long long toff = 0;
    for (const auto& rb : Ri.blk) {
        for (int sp = 0; sp < d; ++sp) {
            if (!usedws[(size_t)rb.w * d + sp]) continue;
            int ia = ba.find(bc.q[rb.k] - qn[sp]);
            if (ia < 0) continue;
            int bbk = S.at(ia, sp);
            if (bbk < 0) continue;
            const auto& BB = S.blk[bbk];
            t1idx[((size_t)rb.i * W.Dr + rb.w) * d + sp] = (int)t1.size();
            t1.push_back({toff, BB.rows, rb.rows});
            const GSeg sg{rb.row * Ri.ld, srow[bbk] * ldS, rb.cols, 0};
            g1.add(rb.rows, BB.rows, toff, Ri.ld, 1, ldS, 1, 1, rb.rows, &sg, 1, 0, 1.0);
            toff += (long long)BB.rows * rb.rows;
        }
    }
    // stage 2: T2(w, s, icb) [a][c_bra] = sum W[w,s,s',w'] T1(icb, w', s')
    const EnvLayout& Ro = Rout.lay;
    const int ldT = pad_ld(bc.maxm(), prec);
    MixList mx;
    std::vector<long long> t2row((size_t)W.Dl * d * bc.n(), -1);
    long long trow = 0;
    for (int w = 0; w < W.Dl; ++w)
        for (int s = 0; s < d; ++s) {
            const std::vector<WE>& we = went[(size_t)w * d + s];
            if (we.empty()) continue;
            for (int icb = 0; icb < bc.n(); ++icb) {
                const int iab = ba.find(bc.q[icb] - qn[s]);
                if (iab < 0 || S.at(iab, s) < 0 || Ro.at(iab, w) < 0) continue;
                const int first = (int)mx.terms.size();
                const TB* x0 = nullptr;
                for (const WE& e : we) {
                    const int ti = t1idx[((size_t)icb * W.Dr + e.wp) * d + e.sp];
                    if (ti < 0) continue;
                    x0 = x0 ? x0 : &t1[ti];
                    mx.terms.push_back({t1[ti].off, t1[ti].cols, 0, e.c});
                }
                if (!x0) continue;
                t2row[((size_t)w * d + s) * bc.n() + icb] = trow;
                MixJob mj{};
                mj.dst = trow * ldT; mj.rows = x0->rows; mj.cols = x0->cols; mj.ldo = ldT;
                mj.zero_to = kpad(x0->cols, prec); mj.t0 = first; mj.nt = (int)mx.terms.size() - first;
                mx.jobs.push_back(mj);
                trow += x0->rows;
            }
        }
    // stage 3: Rout(iab, w) [a_bra][a] = sum_{s, icb} B_s T2(w, s, icb)^T
    GemmBatch g3;
    std::vector<GSeg> sg;
    for (const auto& ob : Ro.blk) {
        sg.clear();
        for (int s = 0; s < d; ++s) {
            int icb = bc.find(ba.q[ob.i] + qn[s]);
            if (icb < 0) continue;
            int bbk = S.at(ob.i, s);
            if (bbk < 0) continue;
            const long long tr = t2row[((size_t)ob.w * d + s) * bc.n() + icb];
            if (tr < 0) continue;
            sg.push_back({tr * ldT, srow[bbk] * ldS, bc.m[icb], 0});
        }
        g3.add(ob.cols, ob.rows, ob.row * Ro.ld, ldT, 1, ldS, 1, 1, Ro.ld, sg);
    }
    stage_env_lists(pk, mx, g1, g3, prec, lists, st);
    DBuf sl, t1b, t2b;
    sl.ensure(std::max<long long>(1, srows) * ldS * num_size(tn), st);
    t1b.ensure(std::max<long long>(1, toff) * num_size(tn), st);
    t2b.ensure(std::max<long long>(1, trow) * ldT * num_size(tn), st);
    run_copy<double>(pk, Bt, sl.p, tn, st);
    run_env_gemm(g1, prec, Rin.buf.p, Ri.rows, Ri.ld, sl.p, srows, ldS, t1b.p, err, st);
    if (tn == Num::F64) run_mix<double>(mx, t1b.as<double>(), t2b.p, tn, st);
    else run_mix<float>(mx, t1b.as<float>(), t2b.p, tn, st);
    run_env_gemm(g3, prec, t2b.p, trow, ldT, sl.p, srows, ldS, Rout.buf.p, err, st);
    Rout.op_valid = false;
    Rout.op32_valid = false;
    PD_CK(cudaStreamSynchronize(st));
}

// ------------------------------------------------------------------------------------------
// Two-site wavefunction from site tensors
// ------------------------------------------------------------------------------------------
void form_two_site(const Sec& bl, const Sec& bm, const Sec& br, const std::vector<int>& qn, const double* left,
                   const double* right, const double* mid, double* psi, cudaStream_t st) {
    const int d = (int)qn.size();
    const SiteLayout SL = site_layout(bl, bm, qn);
    const SiteLayout SR = site_layout(bm, br, qn);
    const PsiLayout P = psi_layout(bl, br, qn);
    DBuf scaled;
    const double* lsrc = left;
    if (mid) {
        // left' = left with its middle (column) index scaled by mid
        std::vector<long long> moff(bm.n() + 1, 0);
        for (int i = 0; i < bm.n(); ++i) moff[i + 1] = moff[i] + bm.m[i];
        std::vector<ColScaleJob> jobs;
        int mx = 1;
        for (const auto& b : SL.blk) {
            jobs.push_back({b.off, b.off, moff[b.j], b.rows, b.cols});
            mx = std::max(mx, b.rows * b.cols);
        }
        DBuf dj;
        upload(dj, jobs, st);
        scaled.ensure(std::max<long long>(1, SL.size) * 8, st);
        if (!jobs.empty()) {
            k_colscale<<<dim3(gridn(mx, 256), (unsigned)jobs.size()), 256, 0, st>>>(dj.as<ColScaleJob>(), left, mid,
                                                                                   scaled.as<double>());
            PD_LAUNCHED();
        }
        lsrc = scaled.as<double>();
        PD_CK(cudaStreamSynchronize(st));
    }
    GemmBatch g;
    for (const auto& b : P.blk) {
        int im = bm.find(bl.q[b.i] + qn[b.s1]);
        if (im < 0) continue;
        int lb = SL.at(b.i, b.s1), rb = SR.at(im, b.s2);
        if (lb < 0 || rb < 0) continue;
        // C(m = c, n = a) = sum_mid right[mid][c] left[a][mid]
        g.add(b.cols, b.rows, b.off, 1, b.cols, bm.m[im], 1, 1, b.cols,
              {GSeg{SR.blk[rb].off, SL.blk[lb].off, bm.m[im], 0}});
    }
    PD_CK(cudaMemsetAsync(psi, 0, sizeof(double) * std::max<long long>(1, P.size), st));
    (void)d;
    run_gemm64(g, right, lsrc, psi, st);
    PD_CK(cudaStreamSynchronize(st));
}

// ------------------------------------------------------------------------------------------
// SVD split with truncation (Eq. svd)
// ------------------------------------------------------------------------------------------
namespace {
struct SecInfo {
    int qm = 0;
    std::map<std::pair<int, int>, int> roff, coff;   // (i, s1) -> row offset, (s2, k) -> col offset
    int r = 0, c = 0;
};
std::map<int, SecInfo> split_sectors(const PsiLayout& P, const Sec& bl, const Sec& br, const std::vector<int>& qn1) {
    std::map<int, SecInfo> secs;
    for (const auto& b : P.blk) {
        int qm = bl.q[b.i] + qn1[b.s1];
        auto& S = secs[qm];
        S.qm = qm;
        S.roff[{b.i, b.s1}] = 0;
        S.coff[{b.s2, b.k}] = 0;
    }
    for (auto& kv : secs) {
        auto& S = kv.second;
        int o = 0;
        for (auto& r : S.roff) { r.second = o; o += bl.m[r.first.first]; }
        S.r = o;
        o = 0;
        for (auto& c : S.coff) { c.second = o; o += br.m[c.first.second]; }
        S.c = o;
    }
    return secs;
}
}  // namespace

void svd_split_bounds(const Sec& bl, const Sec& br, const std::vector<int>& qn1, const std::vector<int>& qn2,
                      long long* a_elems, long long* b_elems, long long* lam_elems) {
    const PsiLayout P = psi_layout2(bl, br, qn1, qn2);
    auto secs = split_sectors(P, bl, br, qn1);
    long long a = 0, b = 0, l = 0;
    for (auto& kv : secs) {
        long long k = std::min(kv.second.r, kv.second.c);
        a += (long long)kv.second.r * k;
        b += k * kv.second.c;
        l += k;
    }
    *a_elems = a;
    *b_elems = b;
    *lam_elems = l;
}

namespace {

// Column copy: dst[dst + r] = scale * src[src + r] for r < rows, scale = 1 / sig[sig_idx] (0 when
// that value is 0) if sig_idx >= 0, else 1.  One CTA per column.
struct ColJob {
    long long src, dst, sig_idx;
    int rows, pad_;
};
__global__ void k_col_copy(const ColJob* __restrict__ jobs, const double* __restrict__ src, double* __restrict__ dst,
                           const double* __restrict__ sig) {
    const ColJob j = jobs[blockIdx.x];
    double sc = 1.0;
    if (j.sig_idx >= 0) {
        const double v = sig[j.sig_idx];
        sc = v > 0.0 ? 1.0 / v : 0.0;
    }
    for (int r = threadIdx.x; r < j.rows; r += blockDim.x) dst[j.dst + r] = sc * src[j.src + r];
}

void col_copy(const std::vector<ColJob>& jobs, const double* src, double* dst, const double* sig, cudaStream_t st) {
    if (jobs.empty()) return;
    DBuf dj;
    upload(dj, jobs, st);
    k_col_copy<<<(unsigned)jobs.size(), 128, 0, st>>>(dj.as<ColJob>(), src, dst, sig);
    PD_LAUNCHED();
}

// FP64 one-sided Jacobi SVD of the column-major matrices W_s (p_s x n_s, n_s <= p_s) at ss[s].w_off
// of W (overwritten by U_s Sigma_s).  Fills v_off / s_off / npad / pair0 of ss; V receives V_s,
// sig the column norms and ord their descending order; dsecs the device copy of ss.
// FP32 block Jacobi (one task per block pair, n / 16 - 1 rounds per sweep) of the batch ss: W (p x n
// at w_off), rotations accumulated into V (n x n at v_off, initialised by the caller); rot: sweep
// histogram (max_sweeps + 1 ints, zeroed), err: error word.  noise_c: the absolute rounding level below
// which a pair is left (times sigma_max; 0: the relative test alone).
void block_jacobi32(const std::vector<SvdSec>& ss, const SvdSec* dsecs, float* W, float* V, int max_rows, int max_sweeps,
                    int* rot, unsigned* err, unsigned long long* flops, cudaStream_t st, float noise_c = 8.0f * FLT_EPSILON) {
    const int nsec = (int)ss.size();
    std::vector<BjSec> bs(nsec);
    std::vector<int> task_sec;
    int nrounds = 0, nblk = 0, npst = 0;
    for (int s = 0; s < nsec; ++s) {
        BjSec b{};
        b.nb = (ss[s].n + 15) / 16;
        b.nbp = b.nb + (b.nb & 1);
        b.task0 = (int)task_sec.size();
        b.ntask = b.nb == 0 ? 0 : (b.nb == 1 ? 1 : b.nbp / 2);
        // each sector's own threshold, so a split's result does not depend on its batch
        b.tol = std::max(3e-5f, 16.0f * FLT_EPSILON * std::sqrt((float)std::max(1, ss[s].p)));
        b.blk0 = nblk;
        b.pst0 = npst;
        nblk += b.nb;
        npst += b.nb * b.nb;
        for (int t = 0; t < b.ntask; ++t) task_sec.push_back(s);
        if (b.nb > 0) nrounds = std::max(nrounds, b.nb == 1 ? 1 : b.nbp - 1);
        bs[s] = b;
    }
    // the dependency queue's items for one sweep: round by round, in each round the pairs of every
    // sector that has the round, taller sectors first (their pairs are the longest)
    std::vector<int> by_rows(nsec);
    for (int s = 0; s < nsec; ++s) by_rows[s] = s;
    std::stable_sort(by_rows.begin(), by_rows.end(), [&](int a, int b) { return ss[a].p > ss[b].p; });
    std::vector<int2> items;
    int nact = 0;
    for (const BjSec& b : bs) nact += b.nb > 0;
    for (int r = 0; r < nrounds; ++r)
        for (int s : by_rows) {
            const BjSec& b = bs[s];
            const int nr = b.nb == 0 ? 0 : (b.nb == 1 ? 1 : b.nbp - 1);
            if (r < nr)
                for (int t = 0; t < b.ntask; ++t) items.push_back(make_int2(s, (r << 16) | t));
        }
    const int bj_sweeps = std::min(40, max_sweeps);   // sweep cap of the block Jacobi
    PD_REQUIRE(nrounds < 32768 && (long long)items.size() * bj_sweeps < (1ll << 31), DMRG_ERR_CAPACITY,
               "block Jacobi: too many work items");
    DBuf dbs, dts, dgmax, dstamp, ditems, dq;
    upload(dbs, bs, st);
    upload(dts, task_sec, st);
    upload(ditems, items, st);
    const size_t nq = 3 + (size_t)nsec * (1 + 2 * bj_sweeps);
    dq.ensure(nq * 4, st);
    PD_CK(cudaMemsetAsync(dq.p, 0, nq * 4, st));
    dgmax.ensure(std::max(1, nsec) * 4, st);
    PD_CK(cudaMemsetAsync(dgmax.p, 0, std::max(1, nsec) * 4, st));
    // block / pair stamps (zero: never rotated / never found converged), the queue's ordering words
    const size_t nstamp = (size_t)std::max(1, 3 * nblk + npst);
    dstamp.ensure(nstamp * 4, st);
    PD_CK(cudaMemsetAsync(dstamp.p, 0, nstamp * 4, st));
    PD_CK(cudaMemsetAsync(flops, 0, 8, st));
    int* stamps = dstamp.as<int>();
    launch_bjacobi(dsecs, dbs.as<BjSec>(), dts.as<int>(), (int)task_sec.size(), nrounds, max_rows, bj_sweeps, W, V,
                   noise_c, dgmax.as<float>(), stamps, stamps + nblk, stamps + nblk + npst, nblk, rot, rot + max_sweeps,
                   err, flops, ditems.as<int2>(), (int)items.size(), nsec, nact, dq.as<int>(), st);
}

// Preconditioning of an FP64 one-sided Jacobi SVD of the batch ss (W FP64, p x n at w_off): the FP32
// block Jacobi on an FP32 copy, its rotations orthonormalised in FP64 (Newton-Schulz) into V
// (n x n at v_off), and W <- W V in FP64.  The FP64 Jacobi then starts from V with columns that are
// orthogonal to FP32 accuracy, so its sweeps converge in the quadratic regime.
void fp64_precondition(const std::vector<SvdSec>& ss, const SvdSec* dsecs, DBuf& dW, double* V, long long woff,
                       long long voff, int maxp, int maxn, unsigned* err, cudaStream_t st) {
    const int max_sweeps = 60;
    DBuf w32, v32, rot32, fl, dW1;
    w32.ensure(woff * 4, st);
    v32.ensure(std::max<long long>(1, voff) * 4, st);
    rot32.ensure((max_sweeps + 1) * 4, st);
    fl.ensure(8, st);
    PD_CK(cudaMemsetAsync(rot32.p, 0, (max_sweeps + 1) * 4, st));
    convert_flat(dW.p, Num::F64, w32.p, Num::F32, woff, st);
    launch_svd_init_v<float>(dsecs, (int)ss.size(), maxn, v32.as<float>(), st);
    block_jacobi32(ss, dsecs, w32.as<float>(), v32.as<float>(), maxp, max_sweeps, rot32.as<int>(), err,
                   fl.as<unsigned long long>(), st);
    convert_flat(v32.p, Num::F32, V, Num::F64, voff, st);
    orthonormalize_square(ss, V, st, 8);          // (from FP32's 1e-4 two or three steps)
    GemmBatch gwq;
    for (const auto& x : ss)
        if (x.n > 0)   // W1(r, c) = sum_u W(r, u) V(u, c)
            gwq.add(x.p, x.n, x.w_off, 1, x.p, x.n, 1, 1, x.p, {GSeg{x.w_off, x.v_off, x.n, 0}});
    dW1.ensure(woff * 8, st);
    run_gemm64(gwq, dW.as<double>(), V, dW1.as<double>(), st);
    dW = std::move(dW1);
}

// ------------------------------------------------------------------------------------------
// FP64 polish of a nearly finished one-sided Jacobi SVD by whole-matrix rotations.
//
// After fp64_precondition the columns of W are orthogonal to FP32 accuracy.  A scalar FP64 Jacobi
// from there costs n - 1 rounds a sweep for some seven sweeps, each round a chain of dot products,
// a reduction, a root and a division on FP64 units that issue 2 DFMA per clock and SM, and a grid
// barrier: 86 ms for the 512-state bond of a chain.  Instead all pairs are rotated at once:
//   G = W^T W;  E(i, j) = -E(j, i) = tan of the Jacobi rotation of the pair (i, j);
//   Q = the orthogonal polar factor of I + E (exactly the Jacobi rotation for a single pair);
//   W <- W Q,  V <- V Q.
// The angles that this leaves are of second order in E, so from 1e-6 two or three passes end at
// rounding level; each is a handful of grouped GEMMs.  The test is the scalar Jacobi's own: no pair
// with |g_ij| > tol |w_i| |w_j|; a batch that has not met it after kPolishPasses goes on with the
// scalar Jacobi.  W and V are updated as W + W (Q - I): the entries of Q - I fall with sigma_j /
// sigma_i, so small columns keep their relative accuracy.
// Columns below about 1e-6 of the largest are not resolved by FP32 at all.  The first pass frees them
// of the large columns (those angles are small) and leaves the angles among themselves, which a second
// FP32 block Jacobi on these columns alone, scaled to order one, then makes small.
// Columns of nearly equal norm want wide angles (tan > 0.1).  Taken beside the small ones these spoil the
// quadratic convergence (what is left of a small angle is then a share of it, not its square), and those
// between exactly degenerate columns are not even wanted: their cosines are the products of those with the
// other columns and vanish with them.  So a pair of nearly equal columns turns only where its cosine is
// above the tolerance and above what the others explain (the root of the product of the two columns' sums of
// squared cosines), and a cluster of five or more columns goes to the scalar Jacobi at once.  A 200 x 200
// matrix of two values: 13.2 ms with all angles taken together (and the scalar Jacobi after), 2.8 now, 14.6
// by the scalar Jacobi alone; 300 values 1e-9 apart, which only that one settles: 57.3, 54.8 and 55.7.
// (Waiting for all small angles instead costs passes where a few pairs are close: 7 to 15 for 5 or 6 at an
// FP64 m = 2000 bond.)
// Columns below kNull of the sector's largest are finished: W V was formed in FP64, so a column that is
// not zero in exact arithmetic does not come out below rounding, 1e-16 of the largest, and one that is (an
// exactly low-rank matrix: its columns are multiples of each other, bit for bit) falls by that factor in
// every pass without ever being orthogonal to its like.  Splits drop such values at 1e-12, gauge moves
// absorb the columns unnormalised.  Without the floor an all-ones 200 x 200 matrix took 95 ms (four passes
// and 60 sweeps of the scalar Jacobi, which has the same floor now), 21 by the scalar Jacobi alone, 1.8 with
// it; integers of rank 3, 200 x 200: 252, 244 and 12 ms.
// Whole splits, at this step: 512-state chain bond 96 -> 31 ms, accurate at the 24x8 cylinder's m = 1000 bond
// 164 -> 52 ms, and closer to 64 bits than the scalar Jacobi's (2.8e-15 against 1.8e-14).
// ------------------------------------------------------------------------------------------
constexpr int kPolishPasses = 16;
constexpr double kNull = 0x1p-80;             // 8e-25, in column norms
constexpr double kClose = 1e-5;               // relative distance of two squared norms

// One CTA per column j of a sector: E(:, j) from the lower triangle of G (rows i >= 64 (j / 64)).  Pairs above
// tol / 10 turn, close ones (see above) only above tol, and those are left to k_polish_take, as sign (2 + t).
// cos2: the column's sum of squared cosines with the columns not close to it.  stat, four words per sector:
// [0] columns with a pair above tol, [1] n - (first column of an unresolved pair: cos > 1e-3 and tan > 0.1),
// [2] largest squared norm of a column of E without the close pairs, as float bits, [3] nonzero: there are
// close pairs above tol.
// A pair costs two roots and three divisions on the FP64 units, 1 to 2 ms a launch at an m = 2000 bond:
// what depends on its result (the cut, the close pairs) reads E instead of working it out again.
struct PolCol {
    int sec, j;
};
__global__ void __launch_bounds__(128)
    k_polish_angles(const SvdSec* __restrict__ secs, const PolCol* __restrict__ cols, const double* __restrict__ G,
                    double* __restrict__ E, float* __restrict__ cos2, unsigned* __restrict__ stat, int nshared) {
    extern __shared__ double diag[];               // G's diagonal, for sectors of up to nshared columns
    const PolCol pc = cols[blockIdx.x];
    const SvdSec s = secs[pc.sec];
    const int j = pc.j, n = s.n;
    const double* Gs = G + s.v_off;
    double* Ej = E + s.v_off + (long long)j * n;
    const double gjj = Gs[j + (long long)j * n];
    const double tol = 4.0 * DBL_EPSILON * sqrt((double)s.p);
    // squared norms are not negative: they order like their bits (NaN above all, and no floor then)
    __shared__ long long tops[4];
    long long top = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double gii = Gs[i + (long long)i * n];
        top = max(top, __double_as_longlong(gii));
        if (n <= nshared) diag[i] = gii;
    }
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((threadIdx.x & 31) == 0) tops[threadIdx.x >> 5] = top;
    __syncthreads();
    const double null2 = kNull * kNull * __longlong_as_double(max(max(tops[0], tops[1]), max(tops[2], tops[3])));
    const double rjj = sqrt(gjj);
    float sum = 0.f, csum = 0.f;
    int above = 0, first = n, close = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int lo = min(i, j), hi = max(i, j);
        const double g = Gs[hi + (long long)lo * n], gii = n <= nshared ? diag[i] : Gs[i + (long long)i * n];
        double t = 0.0;
        const double size = sqrt(gii) * rjj;
        if (i != j && fabs(g) > 0.1 * tol * size && !(fmin(gii, gjj) <= null2)) {
            const bool over = fabs(g) > tol * size;
            above |= over;
            const double zeta = (gjj - gii) / (2.0 * g);
            t = 1.0 / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
            if (t > 0.1 && fabs(g) > 1e-3 * size) first = min(first, lo);
            if (t > 0.1 || fabs(gjj - gii) <= kClose * fmax(gii, gjj)) {
                close |= over;
                t = over ? 2.0 + t : 0.0;
            } else {
                const float c = (float)(fabs(g) / size);
                csum = fmaf(c, c, csum);
                sum = fmaf((float)t, (float)t, sum);
            }
            if (zeta < 0.0 || (zeta == 0.0 && i > j)) t = -t;
        }
        Ej[i] = t;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        csum += __shfl_xor_sync(0xffffffffu, csum, o);
        first = min(first, __shfl_xor_sync(0xffffffffu, first, o));
    }
    above = __any_sync(0xffffffffu, above);
    close = __any_sync(0xffffffffu, close);
    __shared__ float ssum[4], scos[4];
    if ((threadIdx.x & 31) == 0) {
        ssum[threadIdx.x >> 5] = sum;
        scos[threadIdx.x >> 5] = csum;
        if (above) atomicAdd(&stat[4 * pc.sec], 1u);
        if (first < n) atomicMax(&stat[4 * pc.sec + 1], (unsigned)(n - first));
        if (close) atomicOr(&stat[4 * pc.sec + 3], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&stat[4 * pc.sec + 2], __float_as_uint(ssum[0] + ssum[1] + ssum[2] + ssum[3]));
        cos2[s.s_off + j] = scos[0] + scos[1] + scos[2] + scos[3];
    }
}

// What of E turns: no pair of two columns at or after cut[sector]; a close pair, by tan = 0.6 at most, where
// its cosine is above 1.5 times what the others explain.  norms, two words per sector (float bits): largest
// squared norm of a column of E without the close pairs and with them.
__global__ void __launch_bounds__(128)
    k_polish_take(const SvdSec* __restrict__ secs, const PolCol* __restrict__ cols, const double* __restrict__ G,
                  double* __restrict__ E, const int* __restrict__ cut, const float* __restrict__ cos2,
                  unsigned* __restrict__ norms) {
    const PolCol pc = cols[blockIdx.x];
    const SvdSec s = secs[pc.sec];
    const int j = pc.j, n = s.n, from = cut[pc.sec];
    const double* Gs = G + s.v_off;
    double* Ej = E + s.v_off + (long long)j * n;
    cos2 += s.s_off;
    float narrow = 0.f, all = 0.f;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double e = Ej[i];
        double t = e;
        const int lo = min(i, j), hi = max(i, j);
        if (lo >= from) {
            t = 0.0;
        } else if (fabs(e) > 1.0) {
            const double c = fabs(Gs[hi + (long long)lo * n]) /
                             (sqrt(Gs[lo + (long long)lo * n]) * sqrt(Gs[hi + (long long)hi * n]));
            t = c > (double)(1.5f * sqrtf(cos2[i] * cos2[j])) ? copysign(fmin(fabs(e) - 2.0, 0.6), e) : 0.0;
            all = fmaf((float)t, (float)t, all);
        } else {
            narrow = fmaf((float)t, (float)t, narrow);
        }
        if (t != e) Ej[i] = t;
    }
    for (int o = 16; o > 0; o >>= 1) {
        narrow += __shfl_xor_sync(0xffffffffu, narrow, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    __shared__ float sn[4], sa[4];
    if ((threadIdx.x & 31) == 0) {
        sn[threadIdx.x >> 5] = narrow;
        sa[threadIdx.x >> 5] = all;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        narrow = (sn[0] + sn[1]) + (sn[2] + sn[3]);
        all = narrow + ((sa[0] + sa[1]) + (sa[2] + sa[3]));
        atomicMax(&norms[2 * pc.sec], __float_as_uint(narrow));
        atomicMax(&norms[2 * pc.sec + 1], __float_as_uint(all));
    }
}

// X = scale E + a I over the sectors' n x n matrices (X may be E).
__global__ void k_polish_shift(const SvdSec* __restrict__ secs, const PolCol* __restrict__ cols, const double* E,
                               double scale, double a, double* X) {
    const PolCol pc = cols[blockIdx.x];
    const SvdSec s = secs[pc.sec];
    const long long o = s.v_off + (long long)pc.j * s.n;
    for (int i = threadIdx.x; i < s.n; i += blockDim.x) X[o + i] = fma(scale, E[o + i], i == pc.j ? a : 0.0);
}

// Returns true when every pair of columns meets the tolerance (*passes: passes taken).
bool polish64(const std::vector<SvdSec>& ss, const SvdSec* dsecs, DBuf& dW, DBuf& dV, long long woff, long long voff,
              long long soff, unsigned* err, int* passes, cudaStream_t st) {
    const int nsec = (int)ss.size();
    std::vector<PolCol> cols;
    GemmBatch gG, gW, gV, gE;
    gG.repeated = gW.repeated = gV.repeated = true;    // once a pass, five to ten passes
    for (int s = 0; s < nsec; ++s) {
        const SvdSec& x = ss[s];
        for (int j = 0; j < x.n; ++j) cols.push_back({s, j});
        add_gram(gG, x.n, x.v_off, x.p, 1, {GSeg{x.w_off, x.w_off, x.p, 0}});
        gW.add(x.p, x.n, x.w_off, 1, x.p, x.n, 1, 1, x.p, {GSeg{x.w_off, x.v_off, x.n, 0}}, 1);
        gV.add(x.n, x.n, x.v_off, 1, x.n, x.n, 1, 1, x.n, {GSeg{x.v_off, x.v_off, x.n, 0}}, 1);
        gE.add(x.n, x.n, x.v_off, 1, x.n, x.n, 1, 1, x.n, {GSeg{x.v_off, x.v_off, x.n, 0}}, 1, 0.5);
    }
    *passes = 0;
    if (cols.empty()) return true;
    DBuf dcols, G, E, X, Wn, Vn, norms, cos2, stat;
    upload(dcols, cols, st);
    G.ensure(voff * 8, st);
    E.ensure(voff * 8, st);
    X.ensure(voff * 8, st);
    Wn.ensure(woff * 8, st);
    Vn.ensure(voff * 8, st);
    norms.ensure(soff * 8, st);
    cos2.ensure(soff * 4, st);
    stat.ensure((size_t)nsec * 24, st);
    std::vector<unsigned> hs((size_t)nsec * 4);
    std::vector<double> hd(soff);
    const unsigned nc = (unsigned)cols.size();
    std::vector<int> cut(nsec);
    DBuf dcut;
    int maxn = 1;
    for (const SvdSec& x : ss) maxn = std::max(maxn, x.n);
    const int nshared = std::min(maxn, 4096);
    int large = 0;                        // passes whose wide angles were large together
    int stages = 3;                       // FP32 passes over unresolved columns still allowed
    // false: too far from orthogonal; W and V are as before, for the scalar Jacobi to go on with
    auto orthonormalized = [&](const std::vector<SvdSec>& of, DBuf& Q, int steps) {
        try {
            return orthonormalize_square(of, Q.as<double>(), st, steps);
        } catch (const Error& e) {
            if (e.st != DMRG_ERR_NUMERIC) throw;
            return false;
        }
    };
    for (int pass = 0; pass < kPolishPasses; ++pass) {
        run_gemm64(gG, dW.as<double>(), dW.as<double>(), G.as<double>(), st);
        PD_CK(cudaMemsetAsync(stat.p, 0, (size_t)nsec * 24, st));
        k_polish_angles<<<nc, 128, (size_t)nshared * 8, st>>>(dsecs, dcols.as<PolCol>(), G.as<double>(), E.as<double>(),
                                                              cos2.as<float>(), stat.as<unsigned>(), nshared);
        PD_LAUNCHED();
        PD_CK(cudaMemcpyAsync(hs.data(), stat.p, (size_t)nsec * 16, cudaMemcpyDeviceToHost, st));
        PD_CK(cudaStreamSynchronize(st));
        bool unresolved = false, above = false, close = false, finite = true;
        for (int s = 0; s < nsec; ++s) {
            above = above || hs[4 * s] > 0;
            unresolved = unresolved || (stages > 0 && hs[4 * s + 1] > 0);
            close = close || hs[4 * s + 3] > 0;
        }
        if (!above) return true;
        *passes = pass + 1;
        auto largest = [&](int first, int step) {          // of squared norms
            float m = 0.f;
            for (int s = 0; s < nsec; ++s) {
                float v;
                std::memcpy(&v, &hs[first + step * s], 4);
                finite = finite && std::isfinite(v);
                m = std::max(m, std::sqrt(v));
            }
            return m;
        };
        float narrow = largest(2, 4), norm = narrow;       // of E without close pairs, and with them
        if (unresolved || close) {
            // the unresolved columns turn against the others only
            for (int s = 0; s < nsec; ++s) cut[s] = ss[s].n - (unresolved ? (int)hs[4 * s + 1] : 0);
            upload(dcut, cut, st);
            unsigned* norms2 = stat.as<unsigned>() + 4 * nsec;
            k_polish_take<<<nc, 128, 0, st>>>(dsecs, dcols.as<PolCol>(), G.as<double>(), E.as<double>(), dcut.as<int>(),
                                              cos2.as<float>(), norms2);
            PD_LAUNCHED();
            PD_CK(cudaMemcpyAsync(hs.data(), norms2, (size_t)nsec * 8, cudaMemcpyDeviceToHost, st));
            PD_CK(cudaStreamSynchronize(st));
            narrow = largest(0, 2);
            norm = largest(1, 2);
            // columns that all want large angles among themselves do not settle this way
            if (close && norm > 0.6f && !unresolved && (norm > 1.2f || ++large > 2)) return false;
        }
        if (!finite) return false;
        // E <- Q - I
        if (norm <= 1e-6f) {
            // (I + E)(I - E^2)^(-1/2) = I + E + E^2 / 2 + O(|E|^3)
            PD_CK(cudaMemcpyAsync(X.p, E.p, voff * 8, cudaMemcpyDeviceToDevice, st));
            run_gemm64(gE, E.as<double>(), E.as<double>(), X.as<double>(), st);
            std::swap(E, X);
        } else {
            k_polish_shift<<<nc, 128, 0, st>>>(dsecs, dcols.as<PolCol>(), E.as<double>(), norm > 0.6f ? 0.6 / norm : 1.0,
                                               1.0, X.as<double>());
            PD_LAUNCHED();
            if (!orthonormalized(ss, X, 14)) return false;     // angles too large to take together
            k_polish_shift<<<nc, 128, 0, st>>>(dsecs, dcols.as<PolCol>(), X.as<double>(), 1.0, -1.0, E.as<double>());
            PD_LAUNCHED();
        }
        PD_CK(cudaMemcpyAsync(Wn.p, dW.p, woff * 8, cudaMemcpyDeviceToDevice, st));
        PD_CK(cudaMemcpyAsync(Vn.p, dV.p, voff * 8, cudaMemcpyDeviceToDevice, st));
        run_gemm64(gW, dW.as<double>(), E.as<double>(), Wn.as<double>(), st);
        run_gemm64(gV, dV.as<double>(), E.as<double>(), Vn.as<double>(), st);
        std::swap(dW, Wn);
        std::swap(dV, Vn);
        // FP32 block Jacobi on the columns from the cut of every sector that has unresolved pairs, once the
        // rotations against the resolved columns have become small
        if (!unresolved || narrow > 0.05f) continue;
        --stages;
        launch_svd_norms<double>(dsecs, nsec, maxn, dW.as<double>(), norms.as<double>(), st);
        PD_CK(cudaMemcpyAsync(hd.data(), norms.p, (size_t)soff * 8, cudaMemcpyDeviceToHost, st));
        PD_CK(cudaStreamSynchronize(st));
        std::vector<SvdSec> sub;
        CopyList down;
        GemmBatch gw, gv;
        long long wo = 0, vo = 0;
        int mp = 1, mn = 1;
        for (int s = 0; s < nsec; ++s) {
            if (cut[s] >= ss[s].n) continue;
            const SvdSec& x = ss[s];
            SvdSec y{};
            y.p = x.p;
            y.n = x.n - cut[s];
            y.npad = y.n + (y.n & 1);
            y.w_off = wo;
            y.v_off = vo;
            double top = 0.0;
            for (int j = cut[s]; j < x.n; ++j) top = std::max(top, hd[x.s_off + j]);
            CopyJob j{};
            j.src = x.w_off + (long long)cut[s] * x.p; j.dst = wo; j.rows = y.n; j.cols = x.p;
            j.srs = x.p; j.scs = 1; j.drs = x.p; j.dcs = 1; j.zero_to = 0;
            j.scale = top > 0.0 && std::isfinite(top) ? std::ldexp(1.0, -std::max(-1000, std::ilogb(top))) : 1.0;
            down.add(j);
            const long long wc = x.w_off + (long long)cut[s] * x.p, vc = x.v_off + (long long)cut[s] * x.n;
            gw.add(x.p, y.n, wc, 1, x.p, y.n, 1, 1, x.p, {GSeg{wc, vo, y.n, 0}});
            gv.add(x.n, y.n, vc, 1, x.n, y.n, 1, 1, x.n, {GSeg{vc, vo, y.n, 0}});
            wo += (long long)y.p * y.n;
            vo += (long long)y.n * y.n;
            mp = std::max(mp, y.p);
            mn = std::max(mn, y.n);
            sub.push_back(y);
        }
        const int max_sweeps = 60;
        DBuf w64, w32, v32, v64, rot32, fl, dsub;
        w64.ensure(wo * 8, st);
        w32.ensure(wo * 4, st);
        v32.ensure(vo * 4, st);
        v64.ensure(vo * 8, st);
        rot32.ensure((max_sweeps + 1) * 4, st);
        fl.ensure(8, st);
        upload(dsub, sub, st);
        down.up(st);
        PD_CK(cudaMemsetAsync(rot32.p, 0, (max_sweeps + 1) * 4, st));
        // scaled before the conversion: the columns may lie below what FP32 can hold
        run_copy<double>(down, dW.as<double>(), w64.p, Num::F64, st);
        convert_flat(w64.p, Num::F64, w32.p, Num::F32, wo, st);
        launch_svd_init_v<float>(dsub.as<SvdSec>(), (int)sub.size(), mn, v32.as<float>(), st);
        block_jacobi32(sub, dsub.as<SvdSec>(), w32.as<float>(), v32.as<float>(), mp, max_sweeps, rot32.as<int>(), err,
                       fl.as<unsigned long long>(), st, 0.0f);
        convert_flat(v32.p, Num::F32, v64.p, Num::F64, vo, st);
        if (!orthonormalized(sub, v64, 8)) return false;
        PD_CK(cudaMemcpyAsync(Wn.p, dW.p, woff * 8, cudaMemcpyDeviceToDevice, st));
        PD_CK(cudaMemcpyAsync(Vn.p, dV.p, voff * 8, cudaMemcpyDeviceToDevice, st));
        run_gemm64(gw, dW.as<double>(), v64.as<double>(), Wn.as<double>(), st);
        run_gemm64(gv, dV.as<double>(), v64.as<double>(), Vn.as<double>(), st);
        std::swap(dW, Wn);
        std::swap(dV, Vn);
    }
    return false;
}

// The FP64 one-sided Jacobi of W from V on (after fp64_precondition, or from the identity in the plain mode):
// the polish where it settles, else the scalar sweeps.  rot: max_sweeps + 1 zeroed ints, the last of which
// gets the passes or sweeps taken; pairs: the sectors' column pairs.  Returns true where the polish did not
// settle.
bool jacobi64_finish(const std::vector<SvdSec>& ss, const SvdSec* dsecs, const DBuf& pairs, int npairs, int maxnpad,
                     int max_sweeps, DBuf& dW, DBuf& dV, long long woff, long long voff, long long soff, int* rot,
                     unsigned* bar, unsigned* err, cudaStream_t st) {
    const bool polish = g_svd_qr && woff > 0;
    int passes = 0;
    if (polish && polish64(ss, dsecs, dW, dV, woff, voff, soff, err, &passes, st)) {
        PD_CK(cudaMemcpyAsync(rot + max_sweeps, &passes, sizeof(int), cudaMemcpyHostToDevice, st));
        return false;
    }
    DBuf floor2;
    if (polish) floor2.ensure(std::max<size_t>(1, ss.size()) * 8, st);
    launch_jacobi<double>(dsecs, (int)ss.size(), pairs.as<int>(), npairs, maxnpad, max_sweeps, dW.as<double>(),
                          dV.as<double>(), 4.0 * DBL_EPSILON, polish ? kNull : 0.0, floor2.as<double>(), rot,
                          rot + max_sweeps, bar, err, st);
    return polish;
}

void jacobi64(std::vector<SvdSec>& ss, DBuf& dWbuf, DBuf& dsecs, DBuf& dV, DBuf& dsig, DBuf& dord, cudaStream_t st) {
    const int nsec = (int)ss.size();
    std::vector<int> pair_sec;
    long long voff = 0, soff = 0;
    int maxn = 0, maxnpad = 0, maxp = 1;
    for (int s = 0; s < nsec; ++s) {
        SvdSec& x = ss[s];
        x.npad = x.n + (x.n & 1);
        x.v_off = voff;
        x.s_off = soff;
        x.pair0 = (int)pair_sec.size();
        for (int i = 0; i < x.npad / 2; ++i) pair_sec.push_back(s);
        voff += (long long)x.n * x.n;
        soff += x.n;
        maxn = std::max(maxn, x.n);
        maxp = std::max(maxp, x.p);
        maxnpad = std::max(maxnpad, x.npad);
    }
    const int max_sweeps = 60;
    DBuf dpairs, drot, dbar;
    upload(dsecs, ss, st);
    upload(dpairs, pair_sec, st);
    dV.ensure(std::max<long long>(1, voff) * 8, st);
    dsig.ensure(std::max<long long>(1, soff) * 8, st);
    dord.ensure(std::max<long long>(1, soff) * 4, st);
    drot.ensure((max_sweeps + 1) * 4, st);
    dbar.ensure(4 * sizeof(unsigned), st);
    PD_CK(cudaMemsetAsync(drot.p, 0, (max_sweeps + 1) * 4, st));
    PD_CK(cudaMemsetAsync(dbar.p, 0, 4 * sizeof(unsigned), st));
    unsigned* bar = dbar.as<unsigned>();
    const long long woff = ss.empty() ? 0 : ss.back().w_off + (long long)ss.back().p * ss.back().n;
    if (g_svd_qr && woff > 0)
        fp64_precondition(ss, dsecs.as<SvdSec>(), dWbuf, dV.as<double>(), woff, voff, maxp, maxn, bar + 3, st);
    else
        launch_svd_init_v<double>(dsecs.as<SvdSec>(), nsec, maxn, dV.as<double>(), st);
    jacobi64_finish(ss, dsecs.as<SvdSec>(), dpairs, (int)pair_sec.size(), maxnpad, max_sweeps, dWbuf, dV, woff, voff, soff,
                    drot.as<int>(), bar, bar + 3, st);
    double* W = dWbuf.as<double>();
    launch_svd_finish<double>(dsecs.as<SvdSec>(), nsec, maxn, W, dsig.as<double>(), dord.as<int>(), st);
    unsigned err = 0;
    PD_CK(cudaMemcpyAsync(&err, bar + 3, 4, cudaMemcpyDeviceToHost, st));
    PD_CK(cudaStreamSynchronize(st));
    PD_REQUIRE(!(err & ERRBIT_TIMEOUT), DMRG_ERR_TIMEOUT, "Jacobi SVD grid barrier timed out");
}

// The Appendix's accurate SVD, applied to a finished batch (W = U Sigma, V, sig, ord; M the
// matrices the SVD was taken of, same layout as W).  Per matrix, with singular values
// lambda_1 >= ... >= lambda_n: p = the first index with lambda_p / lambda_1 < eps; if there is one,
// X = U_p^T M V_p over the columns p..n, the same SVD and refinement recursively on X, then
// U_p <- U_p U_X, V_p <- V_p V_X, lambda_p.. <- lambda_X.  Results written back into W, V, and
// sig / ord recomputed.  top: the largest singular value of the matrix each of ss descends from.  A
// block at its rounding level holds nothing that the split keeps (its cutoff is 1e-12), and the
// rounding noise of an exactly low-rank matrix is of low rank itself, level after level: it is not
// refined (all-ones 200 x 200: 111 ms with all its levels).
constexpr double ACC_EPS = 1e-4;
void accurate_refine(const std::vector<SvdSec>& ss, const SvdSec* dsecs, double* W, double* V, double* sig, int* ord,
                     const double* M, int depth, cudaStream_t st, const std::vector<double>& top = {}) {
    const int nsec = (int)ss.size();
    long long total = 0;
    for (const auto& x : ss) total = std::max(total, x.s_off + x.n);
    if (total == 0) return;
    std::vector<double> hsig(total);
    std::vector<int> hord(total);
    PD_CK(cudaMemcpyAsync(hsig.data(), sig, total * 8, cudaMemcpyDeviceToHost, st));
    PD_CK(cudaMemcpyAsync(hord.data(), ord, total * 4, cudaMemcpyDeviceToHost, st));
    PD_CK(cudaStreamSynchronize(st));
    struct Ref {
        int s, p, q;
        long long up, vp, x;
    };
    std::vector<Ref> refs;
    std::vector<double> xtop;
    long long nup = 0, nvp = 0, nx = 0;
    for (int s = 0; s < nsec; ++s) {
        const SvdSec& S = ss[s];
        if (S.n <= 1) continue;
        const double l0 = hsig[S.s_off + hord[S.s_off]];
        if (!(l0 > 0.0)) continue;
        const double l_top = depth > 0 ? top[s] : l0;
        int p = -1;
        for (int i = 1; i < S.n; ++i)
            if (hsig[S.s_off + hord[S.s_off + i]] / l0 < ACC_EPS) {
                p = i;
                break;
            }
        if (p < 0 || hsig[S.s_off + hord[S.s_off + p]] <= DBL_EPSILON * l_top) continue;
        const int q = S.n - p;
        refs.push_back({s, p, q, nup, nvp, nx});
        xtop.push_back(l_top);
        nup += (long long)S.p * q;
        nvp += (long long)S.n * q;
        nx += (long long)q * q;
    }
    if (refs.empty()) return;
    PD_REQUIRE(depth < 64, DMRG_ERR_NUMERIC, "accurate SVD recursion did not terminate");
    DBuf dUp, dVp, dT, dX;
    dUp.ensure(nup * 8, st);
    dVp.ensure(nvp * 8, st);
    dT.ensure(nup * 8, st);
    dX.ensure(nx * 8, st);
    // U_p (normalised columns of W in descending order from p) and V_p
    std::vector<ColJob> gu, gv;
    for (const auto& r : refs) {
        const SvdSec& S = ss[r.s];
        for (int j = 0; j < r.q; ++j) {
            const int c = hord[S.s_off + r.p + j];
            gu.push_back({S.w_off + (long long)c * S.p, r.up + (long long)j * S.p, S.s_off + c, S.p, 0});
            gv.push_back({S.v_off + (long long)c * S.n, r.vp + (long long)j * S.n, -1, S.n, 0});
        }
    }
    col_copy(gu, W, dUp.as<double>(), sig, st);
    col_copy(gv, V, dVp.as<double>(), nullptr, st);
    // T = M V_p (p x q), X = U_p^T T (q x q)
    GemmBatch g1, g2;
    for (const auto& r : refs) {
        const SvdSec& S = ss[r.s];
        g1.add(S.p, r.q, r.up, 1, S.p, S.n, 1, 1, S.p, {GSeg{S.w_off, r.vp, S.n, 0}});
        g2.add(r.q, r.q, r.x, S.p, 1, S.p, 1, 1, r.q, {GSeg{r.up, r.up, S.p, 0}});
    }
    run_gemm64(g1, M, dVp.as<double>(), dT.as<double>(), st);
    run_gemm64(g2, dUp.as<double>(), dT.as<double>(), dX.as<double>(), st);
    // the same SVD and refinement of X
    std::vector<SvdSec> xs(refs.size());
    for (size_t i = 0; i < refs.size(); ++i) {
        xs[i] = SvdSec{};
        xs[i].w_off = refs[i].x;
        xs[i].p = xs[i].n = refs[i].q;
    }
    DBuf dXW, dXsecs, dXV, dXsig, dXord;
    dXW.ensure(nx * 8, st);
    PD_CK(cudaMemcpyAsync(dXW.p, dX.p, nx * 8, cudaMemcpyDeviceToDevice, st));
    jacobi64(xs, dXW, dXsecs, dXV, dXsig, dXord, st);
    accurate_refine(xs, dXsecs.as<SvdSec>(), dXW.as<double>(), dXV.as<double>(), dXsig.as<double>(),
                    dXord.as<int>(), dX.as<double>(), depth + 1, st, xtop);
    std::vector<int> hxo(nx > 0 ? (size_t)std::max<long long>(1, xs.back().s_off + xs.back().n) : 1);
    PD_CK(cudaMemcpyAsync(hxo.data(), dXord.p, hxo.size() * 4, cudaMemcpyDeviceToHost, st));
    PD_CK(cudaStreamSynchronize(st));
    // X factors with columns in descending order (W_X keeps U_X Sigma_X)
    DBuf dWxp, dVxp;
    dWxp.ensure(nx * 8, st);
    dVxp.ensure(nx * 8, st);
    std::vector<ColJob> gw, gx;
    for (size_t i = 0; i < refs.size(); ++i) {
        const int q = refs[i].q;
        for (int j = 0; j < q; ++j) {
            const int c = hxo[xs[i].s_off + j];
            gw.push_back({xs[i].w_off + (long long)c * q, refs[i].x + (long long)j * q, -1, q, 0});
            gx.push_back({xs[i].v_off + (long long)c * q, refs[i].x + (long long)j * q, -1, q, 0});
        }
    }
    col_copy(gw, dXW.as<double>(), dWxp.as<double>(), nullptr, st);
    col_copy(gx, dXV.as<double>(), dVxp.as<double>(), nullptr, st);
    // new columns: U_p (U_X Sigma_X) into T, V_p V_X into Vn
    DBuf dVn;
    dVn.ensure(nvp * 8, st);
    GemmBatch g3, g4;
    for (const auto& r : refs) {
        const SvdSec& S = ss[r.s];
        g3.add(S.p, r.q, r.up, 1, S.p, r.q, 1, 1, S.p, {GSeg{r.up, r.x, r.q, 0}});
        g4.add(S.n, r.q, r.vp, 1, S.n, r.q, 1, 1, S.n, {GSeg{r.vp, r.x, r.q, 0}});
    }
    run_gemm64(g3, dUp.as<double>(), dWxp.as<double>(), dT.as<double>(), st);
    run_gemm64(g4, dVp.as<double>(), dVxp.as<double>(), dVn.as<double>(), st);
    std::vector<ColJob> sw, sv;
    for (const auto& r : refs) {
        const SvdSec& S = ss[r.s];
        for (int j = 0; j < r.q; ++j) {
            const int c = hord[S.s_off + r.p + j];
            sw.push_back({r.up + (long long)j * S.p, S.w_off + (long long)c * S.p, -1, S.p, 0});
            sv.push_back({r.vp + (long long)j * S.n, S.v_off + (long long)c * S.n, -1, S.n, 0});
        }
    }
    col_copy(sw, dT.as<double>(), W, nullptr, st);
    col_copy(sv, dVn.as<double>(), V, nullptr, st);
    int maxn = 0;
    for (const SvdSec& x : ss) maxn = std::max(maxn, x.n);
    launch_svd_finish<double>(dsecs, nsec, maxn, W, sig, ord, st);
}

}  // namespace

std::vector<SplitResult> svd_split_batch(const std::vector<SplitReq>& reqs, bool accurate, bool fp32, cudaStream_t st) {
    const size_t es = fp32 ? 4 : 8;
    const int nreq = (int)reqs.size();
    // per bond: sector layout (rows (i, s1) sorted, cols (s2, k) sorted, per middle charge); the
    // sectors of all bonds are numbered consecutively and packed into joint W / V / sigma buffers
    struct Front {
        PsiLayout P;
        std::map<int, SecInfo> secs;
        std::vector<SecInfo*> order;
        int sec0 = 0, nsec = 0, total = 0, maxp = 1;
        long long sbase = 0;
    };
    std::vector<Front> fr(nreq);
    std::vector<SvdSec> ss;
    std::vector<int> pair_sec;
    long long woff = 0, voff = 0, soff = 0;
    int maxn = 0, maxnpad = 0, maxp = 1, max_total = 1, max_nsec = 1;
    for (int q = 0; q < nreq; ++q) {
        const SplitReq& R = reqs[q];
        Front& F = fr[q];
        F.P = psi_layout2(R.bl, R.br, *R.qn1, *R.qn2);
        F.secs = split_sectors(F.P, R.bl, R.br, *R.qn1);
        for (auto& kv : F.secs) F.order.push_back(&kv.second);
        F.sec0 = (int)ss.size();
        F.nsec = (int)F.order.size();
        F.sbase = soff;
        for (int s = 0; s < F.nsec; ++s) {
            const auto& S = *F.order[s];
            SvdSec x{};
            x.p = std::max(S.r, S.c);
            x.n = std::min(S.r, S.c);
            x.npad = x.n + (x.n & 1);
            x.w_off = woff; x.v_off = voff; x.s_off = soff;
            x.pair0 = (int)pair_sec.size();
            for (int i = 0; i < x.npad / 2; ++i) pair_sec.push_back(F.sec0 + s);
            woff += (long long)x.p * x.n;
            voff += (long long)x.n * x.n;
            soff += x.n;
            maxn = std::max(maxn, x.n);
            F.maxp = std::max(F.maxp, x.p);
            maxnpad = std::max(maxnpad, x.npad);
            ss.push_back(x);
        }
        F.total = (int)(soff - F.sbase);
        maxp = std::max(maxp, F.maxp);
        max_total = std::max(max_total, F.total);
        max_nsec = std::max(max_nsec, F.nsec);
    }
    const int nsec = (int)ss.size();
    // gather each bond's Psi blocks into its matrices (W = M, or M^T when M is wide; column-major)
    std::vector<CopyList> gather(nreq);
    for (int q = 0; q < nreq; ++q) {
        const Front& F = fr[q];
        const std::vector<int>& qn = *reqs[q].qn1;
        for (const auto& b : F.P.blk) {
            const int qm = reqs[q].bl.q[b.i] + qn[b.s1];
            const int s = (int)(std::find_if(F.order.begin(), F.order.end(), [&](SecInfo* x) { return x->qm == qm; }) -
                                F.order.begin());
            const auto& S = *F.order[s];
            const SvdSec& x = ss[F.sec0 + s];
            const int r0 = S.roff.at({b.i, b.s1}), c0 = S.coff.at({b.s2, b.k});
            CopyJob j{};
            j.src = b.off; j.rows = b.rows; j.cols = b.cols; j.srs = b.cols; j.scs = 1; j.zero_to = 0; j.scale = 1.0;
            if (S.r >= S.c) {
                j.dst = x.w_off + (long long)c0 * S.r + r0; j.drs = 1; j.dcs = S.r;
            } else {
                j.dst = x.w_off + (long long)r0 * S.c + c0; j.drs = S.c; j.dcs = 1;
            }
            gather[q].add(j);
        }
    }
    DBuf dW, dV, dsig, dord, dsecs, dpairs, drot, dkept, dwts, dbar, dflops;
    dflops.ensure(8, st);
    const int max_sweeps = 60;
    dbar.ensure(4 * sizeof(unsigned), st);     // barrier words + the error word
    PD_CK(cudaMemsetAsync(dbar.p, 0, 4 * sizeof(unsigned), st));
    unsigned* bar = dbar.as<unsigned>();
    unsigned* jerr = bar + 3;
    dW.ensure(std::max<long long>(1, woff) * es, st);
    dV.ensure(std::max<long long>(1, voff) * es, st);
    dsig.ensure(std::max<long long>(1, soff) * 8, st);
    dord.ensure(std::max<long long>(1, soff) * 4, st);
    dkept.ensure(std::max(1, nsec) * 4, st);
    dwts.ensure(std::max(1, nreq) * 16, st);
    drot.ensure((max_sweeps + 1) * 4, st);
    upload(dsecs, ss, st);
    upload(dpairs, pair_sec, st);
    for (auto& g : gather) g.up(st);
    PD_CK(cudaMemsetAsync(dW.p, 0, std::max<long long>(1, woff) * es, st));
    PD_CK(cudaMemsetAsync(drot.p, 0, (max_sweeps + 1) * 4, st));
    const int npairs = (int)pair_sec.size();
    cudaEvent_t sv0 = nullptr, sv1 = nullptr;
    if (prof_on()) {
        PD_CK(cudaEventCreate(&sv0));
        PD_CK(cudaEventCreate(&sv1));
        PD_CK(cudaEventRecord(sv0, st));
    }
    // QR preconditioning: the Jacobi runs on X = R^T (n x n per sector, stored at v_off of dV) with
    // its rotations accumulated in dVJ; afterwards dW receives Q [V_J Sigma; 0] and dV the right
    // singular vectors -- the same outputs as the plain Jacobi on W.
    QrPlan qp;
    DBuf dxsecs, dVJ;
    std::vector<SvdSec> xs;
    if (g_svd_qr && woff > 0 && fp32) {
        qp.build<float>(ss, st);
        if (qp.ok) {
            xs = ss;
            for (auto& x : xs) {
                x.w_off = x.v_off;
                x.p = x.n;
            }
            upload(dxsecs, xs, st);
            dVJ.ensure(std::max<long long>(1, voff) * es, st);
        }
    }
    const bool use_qr = qp.ok && !xs.empty();
    const SvdSec* jsecs = use_qr ? dxsecs.as<SvdSec>() : dsecs.as<SvdSec>();
    const int jmaxp = use_qr ? maxn : maxp;
    if (fp32) {
        for (int q = 0; q < nreq; ++q) run_copy<double>(gather[q], reqs[q].psi, dW.p, Num::F32, st);
        float* JW = dW.as<float>();
        float* JV = dV.as<float>();
        if (use_qr) {
            qp.factor<float>(dW.as<float>(), st);
            qp.form_rt<float>(dW.as<float>(), dV.as<float>(), st);
            JW = dV.as<float>();
            JV = dVJ.as<float>();
        }
        launch_svd_init_v<float>(jsecs, nsec, maxn, JV, st);
        // the kept factor that joins a block is re-orthonormalised in FP64 afterwards
        block_jacobi32(use_qr ? xs : ss, jsecs, JW, JV, jmaxp, max_sweeps, drot.as<int>(), jerr,
                       dflops.as<unsigned long long>(), st);
        if (use_qr) {
            DBuf dWo;
            dWo.ensure(std::max<long long>(1, woff) * es, st);
            qp.finish<float>(dW.as<float>(), dV.as<float>(), dVJ.as<float>(), dWo.as<float>(), st);
            dW = std::move(dWo);
        }
        launch_svd_finish<float>(dsecs.as<SvdSec>(), nsec, maxn, dW.as<float>(), dsig.as<double>(), dord.as<int>(), st);
    } else {
        for (int q = 0; q < nreq; ++q) run_copy<double>(gather[q], reqs[q].psi, dW.p, Num::F64, st);
        DBuf dM;
        if (accurate && woff > 0) {
            dM.ensure(woff * 8, st);
            PD_CK(cudaMemcpyAsync(dM.p, dW.p, woff * 8, cudaMemcpyDeviceToDevice, st));
        }
        if (g_svd_qr && woff > 0)
            fp64_precondition(ss, dsecs.as<SvdSec>(), dW, dV.as<double>(), woff, voff, maxp, maxn, jerr, st);
        else
            launch_svd_init_v<double>(dsecs.as<SvdSec>(), nsec, maxn, dV.as<double>(), st);
        if (jacobi64_finish(ss, dsecs.as<SvdSec>(), dpairs, npairs, maxnpad, max_sweeps, dW, dV, woff, voff, soff,
                            drot.as<int>(), bar, jerr, st))
            prof_svd_scalar();
        launch_svd_finish<double>(dsecs.as<SvdSec>(), nsec, maxn, dW.as<double>(), dsig.as<double>(), dord.as<int>(), st);
        if (accurate && woff > 0)
            accurate_refine(ss, dsecs.as<SvdSec>(), dW.as<double>(), dV.as<double>(), dsig.as<double>(),
                            dord.as<int>(), dM.as<double>(), 0, st);
    }
    if (sv0) {
        PD_CK(cudaEventRecord(sv1, st));
        int sweeps = 0;
        unsigned long long fl = 0;
        std::vector<int> hist(max_sweeps, 0);
        PD_CK(cudaMemcpyAsync(&sweeps, drot.as<int>() + max_sweeps, 4, cudaMemcpyDeviceToHost, st));
        PD_CK(cudaMemcpyAsync(hist.data(), drot.p, 4 * max_sweeps, cudaMemcpyDeviceToHost, st));
        if (fp32) PD_CK(cudaMemcpyAsync(&fl, dflops.p, 8, cudaMemcpyDeviceToHost, st));
        PD_CK(cudaStreamSynchronize(st));
        float ms = 0.f;
        PD_CK(cudaEventElapsedTime(&ms, sv0, sv1));
        double alg_fl = 0.0, alg_b = 0.0;
        for (const SvdSec& x : ss) {
            const double p = x.p, n = x.n;
            alg_fl += 4.0 * p * n * n + 22.0 * n * n * n;
            alg_b += 4.0 * (2.0 * p * n + n * n);
        }
        prof_svd(sweeps, ms, fp32 ? 1 : 2, maxp, (double)fl, fp32 ? hist.data() : nullptr, max_sweeps, nreq, alg_fl,
                 alg_b);
        cudaEventDestroy(sv0);
        cudaEventDestroy(sv1);
    }
    // truncation per bond (the keep-m rule runs over one bond's sectors): its sector table with
    // sigma offsets relative to the bond's first sector, and sigma / order shifted to match
    std::vector<SvdSec> tl = ss;
    for (const Front& F : fr)
        for (int s = 0; s < F.nsec; ++s) tl[F.sec0 + s].s_off -= F.sbase;
    DBuf dtl, tsd, tsi;
    upload(dtl, tl, st);
    tsd.ensure((size_t)(max_total + max_nsec + 1) * 8, st);
    tsi.ensure((size_t)(2 * max_total + 1) * 4, st);
    // an FP32 SVD reports exact zeros at ~1e-7 of the largest singular value: keep its cutoff
    // above that noise floor (the discarded weight stays below 1e-10)
    for (int q = 0; q < nreq; ++q) {
        const Front& F = fr[q];
        const double cutoff = fp32 ? std::max(reqs[q].rel_cutoff, 1e-5) : reqs[q].rel_cutoff;
        launch_truncate(dtl.as<SvdSec>() + F.sec0, F.nsec, dsig.as<double>() + F.sbase, dord.as<int>() + F.sbase,
                        F.total, reqs[q].m_max, cutoff, 1e-10, dkept.as<int>() + F.sec0, dwts.as<double>() + 2 * q,
                        tsd.as<double>(), tsi.as<int>(), st);
    }
    std::vector<int> kept(std::max(1, nsec));
    std::vector<double> wts(2 * std::max(1, nreq));
    unsigned jerr_h = 0;
    int sweeps_h = 0;
    PD_CK(cudaMemcpyAsync(&sweeps_h, drot.as<int>() + max_sweeps, 4, cudaMemcpyDeviceToHost, st));
    PD_CK(cudaMemcpyAsync(&jerr_h, jerr, 4, cudaMemcpyDeviceToHost, st));
    PD_CK(cudaMemcpyAsync(kept.data(), dkept.p, 4 * std::max(1, nsec), cudaMemcpyDeviceToHost, st));
    PD_CK(cudaMemcpyAsync(wts.data(), dwts.p, 16 * std::max(1, nreq), cudaMemcpyDeviceToHost, st));
    PD_CK(cudaStreamSynchronize(st));
    PD_REQUIRE(!(jerr_h & ERRBIT_TIMEOUT), DMRG_ERR_TIMEOUT, "Jacobi SVD grid barrier timed out");
    std::vector<SplitResult> out(nreq);
    std::vector<DBuf> keep_alive;
    keep_alive.reserve(4 * nreq);
    for (int q = 0; q < nreq; ++q) {
        const Front& F = fr[q];
        const SplitReq& R = reqs[q];
        const std::vector<int>& qn1 = *R.qn1;
        const std::vector<int>& qn2 = *R.qn2;
        SplitResult& res = out[q];
        res.sweeps = sweeps_h;
        res.max_rows = F.maxp;
        std::vector<int> kept_of_sec(F.nsec, 0);
        for (int s = 0; s < F.nsec; ++s)
            if (kept[F.sec0 + s] > 0) {
                res.mid.q.push_back(F.order[s]->qm);
                res.mid.m.push_back(kept[F.sec0 + s]);
                kept_of_sec[s] = kept[F.sec0 + s];
            }
        PD_REQUIRE(res.mid.n() > 0, DMRG_ERR_NUMERIC, "SVD kept no singular value (zero wavefunction?)");
        const double w0 = wts[2 * q], w1 = wts[2 * q + 1];
        res.trunc = w0 > 0 ? std::max(0.0, (w0 - w1) / w0) : 0.0;
        // scatter
        const SiteLayout SA = site_layout(R.bl, res.mid, qn1);
        const SiteLayout SB = site_layout(res.mid, R.br, qn2);
        std::vector<ScatJob> ja, jb;
        int mx = 1;
        for (int s = 0; s < F.nsec; ++s) {
            if (!kept_of_sec[s]) continue;
            const auto& S = *F.order[s];
            const SvdSec& x = ss[F.sec0 + s];
            const int im = res.mid.find(S.qm);
            const bool rge = S.r >= S.c;
            for (const auto& r : S.roff) {        // A blocks (i, s1) [a][k]
                const int ab = SA.at(r.first.first, r.first.second);
                if (ab < 0) continue;
                ScatJob j{};
                j.dst = SA.blk[ab].off; j.rows = SA.blk[ab].rows; j.cols = SA.blk[ab].cols;
                j.s_off = x.s_off; j.off0 = r.second; j.left = 1; j.lam_pow = R.lam_pow_left;
                if (rge) { j.fromW = 1; j.base = x.w_off; j.ld = x.p; }
                else { j.fromW = 0; j.base = x.v_off; j.ld = x.n; }
                ja.push_back(j);
                mx = std::max(mx, j.rows * j.cols);
            }
            for (const auto& c : S.coff) {        // B blocks (m, s2) [k][c]
                const int bb = SB.at(im, c.first.first);
                if (bb < 0) continue;
                ScatJob j{};
                j.dst = SB.blk[bb].off; j.rows = SB.blk[bb].rows; j.cols = SB.blk[bb].cols;
                j.s_off = x.s_off; j.off0 = c.second; j.left = 0; j.lam_pow = R.lam_pow_right;
                if (rge) { j.fromW = 0; j.base = x.v_off; j.ld = x.n; }
                else { j.fromW = 1; j.base = x.w_off; j.ld = x.p; }
                jb.push_back(j);
                mx = std::max(mx, j.rows * j.cols);
            }
        }
        const double* wq = dwts.as<double>() + 2 * q;
        auto scatter = [&](const std::vector<ScatJob>& jobs_, double* dst) {
            if (jobs_.empty()) return;
            keep_alive.emplace_back();
            DBuf& dj = keep_alive.back();
            upload(dj, jobs_, st);
            dim3 g(gridn(mx, 256), (unsigned)jobs_.size());
            if (fp32)
                k_svd_scatter<float><<<g, 256, 0, st>>>(dj.as<ScatJob>(), dW.as<float>(), dV.as<float>(),
                                                        dsig.as<double>(), dord.as<int>(), wq, dst);
            else
                k_svd_scatter<double><<<g, 256, 0, st>>>(dj.as<ScatJob>(), dW.as<double>(), dV.as<double>(),
                                                         dsig.as<double>(), dord.as<int>(), wq, dst);
            PD_LAUNCHED();
        };
        scatter(ja, R.A_out);
        scatter(jb, R.B_out);
        // lambda
        std::vector<LamJob> lj;
        long long o = 0;
        for (int s = 0; s < F.nsec; ++s) {
            if (!kept_of_sec[s]) continue;
            lj.push_back({ss[F.sec0 + s].s_off, o, kept_of_sec[s], 0});
            o += kept_of_sec[s];
        }
        keep_alive.emplace_back();
        DBuf& dlj = keep_alive.back();
        upload(dlj, lj, st);
        double* lam_dev = R.lam_out_dev;
        if (!lam_dev) {
            keep_alive.emplace_back();
            DBuf& dlam = keep_alive.back();
            dlam.ensure(o * 8, st);
            lam_dev = dlam.as<double>();
        }
        k_lam_out<<<std::max<int>(1, (int)lj.size()), 128, 0, st>>>(dlj.as<LamJob>(), (int)lj.size(),
                                                                     dsig.as<double>(), dord.as<int>(), wq, lam_dev);
        PD_LAUNCHED();
        res.lam.resize(o);
        PD_CK(cudaMemcpyAsync(res.lam.data(), lam_dev, o * 8, cudaMemcpyDeviceToHost, st));
    }
    PD_CK(cudaStreamSynchronize(st));
    return out;
}

SplitResult svd_split(const Sec& bl, const Sec& br, const std::vector<int>& qn1, const std::vector<int>& qn2,
                      const double* psi, int m_max, double rel_cutoff, bool accurate, int lam_pow_left,
                      int lam_pow_right, double* A_out, double* B_out, double* lam_out_dev, cudaStream_t st,
                      bool fp32) {
    SplitReq r;
    r.bl = bl;
    r.br = br;
    r.qn1 = &qn1;
    r.qn2 = &qn2;
    r.psi = psi;
    r.m_max = m_max;
    r.rel_cutoff = rel_cutoff;
    r.lam_pow_left = lam_pow_left;
    r.lam_pow_right = lam_pow_right;
    r.A_out = A_out;
    r.B_out = B_out;
    r.lam_out_dev = lam_out_dev;
    return std::move(svd_split_batch({r}, accurate, fp32, st)[0]);
}

// ------------------------------------------------------------------------------------------
// Davidson (the Sec. II local eigensolver), FP64 vectors, same algorithm as the CPU oracle
// ------------------------------------------------------------------------------------------
DavResult davidson(HeffPlan& P, const EnvSlab& L, const EnvSlab& R, double* x, int kmax, double tol,
                   int max_iter, unsigned* err, cudaStream_t st, HeffPlan* acc, int refine_iters) {
    const long long n = P.psi.size;
    PD_REQUIRE(kmax >= 2 && kmax <= 32, DMRG_ERR_ARG, "Davidson kmax must be in [2, 32]");
    DavResult res;
    DBuf dV, dAV, dG, dyth, dpart, dc, dnrm, du, dAu, dr, dt, ddg, dctr;
    dV.ensure((size_t)kmax * n * 8, st);
    dAV.ensure((size_t)kmax * n * 8, st);
    dG.ensure((size_t)kmax * kmax * 8, st);
    dyth.ensure((kmax + 1) * 8, st);
    dpart.ensure((size_t)2 * kmax * dav_grid(n) * 8, st);
    dc.ensure(2 * kmax * 8, st);
    dnrm.ensure(4 * 8, st);                     // |r|^2, |u|^2, |t|^2, |x|^2
    dctr.ensure(sizeof(unsigned), st);
    du.ensure(n * 8, st);
    dAu.ensure(n * 8, st);
    dr.ensure(n * 8, st);
    dt.ensure(n * 8, st);
    ddg.ensure(n * 8, st);
    PD_CK(cudaMemsetAsync(dctr.p, 0, sizeof(unsigned), st));
    double* V = dV.as<double>();
    double* AV = dAV.as<double>();
    double* G = dG.as<double>();
    double* part = dpart.as<double>();
    double* nrm = dnrm.as<double>();
    unsigned* ctr = dctr.as<unsigned>();
    // pinned, written by kernels: |r|^2, |u|^2, theta, |t|^2
    double* hn = reinterpret_cast<double*>(sweep_flags_host(64));
    constexpr double kFloor = 1e-14;            // a correction this small is rounding
    struct Events {
        cudaStream_t st;
        cudaEvent_t e[4] = {};
        explicit Events(cudaStream_t st_) : st(st_) {
            for (int i = 0; i < 4; ++i)
                PD_CK(i < 2 ? cudaEventCreate(&e[i]) : cudaEventCreateWithFlags(&e[i], cudaEventDisableTiming));
        }
        ~Events() {
            cudaStreamSynchronize(st);           // no kernel writes to hn once this call has left, by throw or return
            for (auto x : e)
                if (x) cudaEventDestroy(x);
        }
    } ev(st);
    HeffPlan* cur = &P;
    // matvec timed by a pair of events, which is read at the next wait (the stream does not stop for it)
    auto mv = [&](const double* in, double* out) {
        PD_CK(cudaEventRecord(ev.e[0], st));
        heff_apply(*cur, L, R, in, out, err, st);
        PD_CK(cudaEventRecord(ev.e[1], st));
    };
    auto mv_done = [&]() {
        float ms = 0.f;
        PD_CK(cudaEventSynchronize(ev.e[1]));
        PD_CK(cudaEventElapsedTime(&ms, ev.e[0], ev.e[1]));
        if (cur == &P) {
            res.mv_ms += ms;
            res.matvecs++;
        } else {
            res.acc_ms += ms;
            res.acc_matvecs++;
        }
    };
    heff_diag(P, L, R, ddg.as<double>(), st);
    // One Davidson run from the vector in x; leaves the Ritz vector in du (|u|^2 in nrm[1]).  The host
    // queues ahead of the stream: the correction vector is made before the residual's norm is read, and
    // the matvec before the correction's norm is (what a stop makes superfluous is a few vector launches
    // or, with an exhausted subspace, a matvec of the zero vector, which is not counted).
    auto run = [&](int iters) {
        launch_dav_norm(x, n, part, ctr, nrm + 3, st);
        launch_dav_unit(x, nrm + 3, 0.0, n, V, st);
        mv(V, AV);
        int k = 1;
        for (int it = 1; it <= iters; ++it) {
            res.iters++;
            launch_dav_gram(V, AV, n, k - 1, kmax, G, part, ctr, true, dyth.as<double>(), st);
            launch_dav_ritz(V, AV, n, k, dyth.as<double>(), du.as<double>(), dAu.as<double>(), dr.as<double>(), part, ctr,
                            nrm, hn, st);
            PD_CK(cudaEventRecord(ev.e[2], st));
            if (it < iters) {
                if (k >= kmax) {   // restart from the Ritz vector
                    launch_dav_unit(du.as<double>(), nrm + 1, 0.0, n, V, st);
                    launch_dav_unit(dAu.as<double>(), nrm + 1, 0.0, n, AV, st);
                    k = 1;
                    launch_dav_gram(V, AV, n, 0, kmax, G, part, ctr, false, nullptr, st);
                }
                launch_dav_correct(V, n, k, dr.as<double>(), ddg.as<double>(), dyth.as<double>(), 1e-4, dt.as<double>(),
                                   dc.as<double>(), dc.as<double>() + kmax, part, ctr, nrm + 2, hn + 3, st);
                launch_dav_unit(dt.as<double>(), nrm + 2, kFloor, n, V + (size_t)k * n, st);
                PD_CK(cudaEventRecord(ev.e[3], st));
            }
            mv_done();
            PD_CK(cudaEventSynchronize(ev.e[2]));
            res.theta = hn[2];
            res.rnorm = std::sqrt(std::max(0.0, hn[0]));
            PD_REQUIRE(std::isfinite(res.theta) && std::isfinite(res.rnorm), DMRG_ERR_NUMERIC,
                       "non-finite Ritz value in Davidson");
            if (res.rnorm <= tol * std::max(1.0, std::fabs(res.theta)) || it == iters) break;
            mv(V + (size_t)k * n, AV + (size_t)k * n);
            PD_CK(cudaEventSynchronize(ev.e[3]));
            if (std::sqrt(hn[3]) < kFloor) break;
            ++k;
        }
        // x = u / |u|
        launch_dav_unit(du.as<double>(), nrm + 1, 0.0, n, x, st);
    };
    run(max_iter);
    if (acc && refine_iters > 0) {
        PD_REQUIRE(acc->psi.size == n, DMRG_ERR_STATE, "refinement plan does not match the bond");
        cur = acc;
        run(refine_iters);
    }
    PD_CK(cudaStreamSynchronize(st));
    return res;
}

}  // namespace pd
