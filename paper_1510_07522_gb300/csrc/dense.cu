// Dense FP64 complex kernels: tiled ZGEMM, bounded grid barrier, one-sided Jacobi.
#include <algorithm>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "dense.cuh"

namespace cg = cooperative_groups;

namespace rsrr {

// ---------------------------------------------------------------------------------------------
// ZGEMM on the FP64 cores.  GB300 issues two FP64 multiply-adds a clock per SM (1.25 TFLOP/s in
// all), so what bounds a product is how evenly its multiply-adds spread over the SMs and their
// sub-partitions, not the operand traffic: a 16 x 16 tile reads one byte a clock.  The tiles are
// therefore small (256 outputs for 128 threads, four warps, two outputs a thread), and K is cut
// over the up to eight CTAs of a cluster, which add their partial tiles through distributed shared
// memory in a fixed order (no atomics, no workspace, the same bits on every run).  The
// FP64 products of one pass (projection and reduced solve), before with 32 x 32 tiles of two warps
// and no K split below 512, and now: n = 9991, k_S = 133: 18.8 -> 3.1 ms; n = 900, moment scheme,
// k_S = 45: 18.5 -> 1.0 ms; n = 5000, k_S = 48, K = 8: 29.7 -> 3.8 ms.
// A tile is 16 x 16, or 64 x 4 for the products with a handful of columns (moments, traces).
// ---------------------------------------------------------------------------------------------
namespace {
constexpr int BK = 16;          // K terms per shared-memory stage
constexpr int kZgThreads = 128;
constexpr int kZgTile = 256;    // outputs per tile
constexpr int kZgMaxSplit = 8;  // portable cluster size

struct ZgOperand {  // op(X)(row, k) = X[row * sr + k * sk], conjugated when conj
    const c128* p;
    int64_t sr, sk, sb;
    int conj;
};
struct ZgArgs {
    ZgOperand A, B;  // B's "row" is the output column
    c128* C;
    int64_t ldc, sC;
    int M, N, K, tm, tn, split, kper;
    c128 alpha, beta;
};

__device__ __forceinline__ c128 zg_fetch(const ZgOperand& o, const c128* base, int r, int R, int k, int k_end) {
    c128 v = czero<double>();
    if (r < R && k < k_end) {
        v = base[r * o.sr + k * o.sk];
        if (o.conj) v.im = -v.im;
    }
    return v;
}

template <int BM, int BN>
__global__ void __launch_bounds__(kZgThreads) zgemm_kernel(ZgArgs g) {
    static_assert(BM * BN == kZgTile, "two outputs a thread");
    constexpr int TX = BN / 2;  // threads across the columns; a thread owns columns tx and tx + TX
    constexpr int NA = BM * BK / kZgThreads, NB = (BN * BK + kZgThreads - 1) / kZgThreads;
    __shared__ c128 As[BK][BM + 1];
    __shared__ c128 Bs[BK][BN + 1];
    __shared__ c128 part[kZgTile];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    // the CTAs of a cluster are the K slices of one tile
    const int64_t tile = blockIdx.x / g.split;
    const int ks = (int)(blockIdx.x % g.split);
    const int bm = (int)(tile % g.tm) * BM, bn = (int)((tile / g.tm) % g.tn) * BN;
    const int64_t b = tile / ((int64_t)g.tm * g.tn);
    const c128* Ab = g.A.p + b * g.A.sb;
    const c128* Bb = g.B.p + b * g.B.sb;
    const int k_begin = min(g.K, ks * g.kper), k_end = min(g.K, k_begin + g.kper);
    // consecutive threads follow whichever index is contiguous in memory
    const bool a_rows = g.A.sr == 1, b_rows = g.B.sr == 1;
    c128 ra[NA], rb[NB];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const int idx = tid + kZgThreads * u;
            const int i = a_rows ? idx % BM : idx / BK, k = a_rows ? idx / BM : idx % BK;
            ra[u] = zg_fetch(g.A, Ab, bm + i, g.M, k0 + k, k_end);
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int idx = tid + kZgThreads * u;
            if (idx < BN * BK) {
                const int j = b_rows ? idx % BN : idx / BK, k = b_rows ? idx / BN : idx % BK;
                rb[u] = zg_fetch(g.B, Bb, bn + j, g.N, k0 + k, k_end);
            }
        }
    };
    c128 acc0 = czero<double>(), acc1 = czero<double>();
    if (k_begin < k_end) fetch(k_begin);
    for (int k0 = k_begin; k0 < k_end; k0 += BK) {
        __syncthreads();  // the previous stage has been read
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const int idx = tid + kZgThreads * u;
            const int i = a_rows ? idx % BM : idx / BK, k = a_rows ? idx / BM : idx % BK;
            As[k][i] = ra[u];
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int idx = tid + kZgThreads * u;
            if (idx < BN * BK) {
                const int j = b_rows ? idx % BN : idx / BK, k = b_rows ? idx / BN : idx % BK;
                Bs[k][j] = rb[u];
            }
        }
        __syncthreads();
        if (k0 + BK < k_end) fetch(k0 + BK);  // in flight under this stage's multiply-adds
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            if (k0 + k >= k_end) break;
            const c128 x = As[k][ty];
            cfma(acc0, x, Bs[k][tx]);
            cfma(acc1, x, Bs[k][tx + TX]);
        }
    }
    auto store = [&](int i, int j, c128 v) {
        const int gi = bm + i, gj = bn + j;
        if (gi >= g.M || gj >= g.N) return;
        c128* c = g.C + b * g.sC + gi + (int64_t)gj * g.ldc;
        v = g.alpha * v;
        *c = (g.beta.re == 0.0 && g.beta.im == 0.0) ? v : v + g.beta * (*c);
    };
    if (g.split == 1) {
        store(ty, tx, acc0);
        store(ty, tx + TX, acc1);
        return;
    }
    part[ty + BM * tx] = acc0;
    part[ty + BM * (tx + TX)] = acc1;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    // the tile's outputs are dealt out over the cluster; each is summed in K order
    for (int e = tid + kZgThreads * ks; e < kZgTile; e += kZgThreads * g.split) {
        c128 v = czero<double>();
        for (int q = 0; q < g.split; ++q) v = v + *cluster.map_shared_rank(&part[e], q);
        store(e % BM, e / BM, v);
    }
    cluster.sync();  // no CTA leaves while its partial tile may still be read
}

__global__ void scale_kernel(c128* C, int M, int N, int64_t ldc, int64_t sC, c128 beta) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int b = blockIdx.y;
    if (idx >= (int64_t)M * N) return;
    const int64_t i = idx % M, j = idx / M;
    c128* c = C + b * sC + i + j * ldc;
    *c = (beta.re == 0.0 && beta.im == 0.0) ? czero<double>() : beta * (*c);
}
}  // namespace

namespace {
ZgOperand zg_operand(const c128* p, int64_t ld, int64_t sb, int op, bool is_b) {
    // A: op(A)(i, k); B is taken by its output column j: op(B)(k, j)
    const bool rows = (op == OP_N) != is_b;  // the row index is the contiguous one
    return ZgOperand{p, rows ? 1 : ld, rows ? ld : 1, sb, op == OP_C ? 1 : 0};
}

template <int BM, int BN>
int zgemm_fp64(const Zgemm& g, cudaStream_t s) {
    ZgArgs a;
    a.A = zg_operand(g.A, g.lda, g.sA, g.opA, false);
    a.B = zg_operand(g.B, g.ldb, g.sB, g.opB, true);
    a.C = g.C; a.ldc = g.ldc; a.sC = g.sC;
    a.M = g.M; a.N = g.N; a.K = g.K;
    a.tm = (int)ceil_div(g.M, BM);
    a.tn = (int)ceil_div(g.N, BN);
    a.alpha = g.alpha; a.beta = g.beta;
    // K slices until every SM has two CTAs, but none shorter than one stage
    const int64_t tiles = (int64_t)a.tm * a.tn * g.batch;
    int split = 1;
    while (split < kZgMaxSplit && tiles * split < 2 * 152 && g.K >= 2 * split * BK) split *= 2;
    a.split = split;
    a.kper = (int)ceil_div(g.K, split);
    if (tiles * split > INT32_MAX) return set_error(RSRR_EINVAL, "zgemm: too many tiles");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * split));
    cfg.blockDim = dim3(kZgThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = split;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    RSRR_CUDA(cudaLaunchKernelEx(&cfg, zgemm_kernel<BM, BN>, a));
    note_launch();
    return RSRR_OK;
}
}  // namespace

// ZGEMM accounting for the calling host thread: device time (events around each call) and
// algorithmic flops 8 M N K per product, between zgemm_profile_begin and zgemm_profile_end.
namespace {
struct ZgemmProfile {
    bool on = false;
    double flops = 0.0, flops_tc = 0.0;
    struct Ev { cudaEvent_t a, b; bool tc; };
    std::vector<Ev> ev;
};
thread_local ZgemmProfile g_zprof;
struct JacobiProfile {
    bool on = false;
    double flops = 0.0;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev;
};
thread_local JacobiProfile g_jprof;
double drain_events(std::vector<std::pair<cudaEvent_t, cudaEvent_t>>& ev) {
    double t = 0.0;
    for (auto& e : ev) {
        float x = 0.f;
        cudaEventSynchronize(e.second);
        cudaEventElapsedTime(&x, e.first, e.second);
        t += x;
        cudaEventDestroy(e.first);
        cudaEventDestroy(e.second);
    }
    ev.clear();
    return t;
}
}  // namespace

void zgemm_profile_begin() {
    g_zprof.on = true;
    g_zprof.flops = g_zprof.flops_tc = 0.0;
    g_zprof.ev.clear();
}

void zgemm_profile_end(double* ms, double* flops, double* ms_tc, double* flops_tc) {
    double t = 0.0, t_tc = 0.0;
    for (auto& e : g_zprof.ev) {
        float x = 0.f;
        cudaEventSynchronize(e.b);
        cudaEventElapsedTime(&x, e.a, e.b);
        t += x;
        if (e.tc) t_tc += x;
        cudaEventDestroy(e.a);
        cudaEventDestroy(e.b);
    }
    g_zprof.ev.clear();
    g_zprof.on = false;
    *ms = t;
    *flops = g_zprof.flops;
    if (ms_tc) *ms_tc = t_tc;
    if (flops_tc) *flops_tc = g_zprof.flops_tc;
}

void jacobi_profile_begin() {
    g_jprof.on = true;
    g_jprof.flops = 0.0;
    g_jprof.ev.clear();
}

void jacobi_profile_end(double* ms, double* flops) {
    *ms = drain_events(g_jprof.ev);
    *flops = g_jprof.flops;
    g_jprof.on = false;
}

static int zgemm_dispatch(const Zgemm& g0, cudaStream_t s);

namespace {
thread_local int g_zpath = 0;
}
void zgemm_set_path(int path) { g_zpath = path; }
int zgemm_get_path() { return g_zpath; }

int zgemm(const Zgemm& g0, cudaStream_t s) {
    if (!g_zprof.on || g0.M <= 0 || g0.N <= 0 || g0.K <= 0 || g0.batch <= 0) return zgemm_dispatch(g0, s);
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, s);
    const int rc = zgemm_dispatch(g0, s);
    cudaEventRecord(b, s);
    const bool tc = g_zpath == 2 || (g_zpath == 0 && !g0.fp64 && zgemm_tc_fits(g0));
    g_zprof.ev.push_back({a, b, tc});
    const double f = 8.0 * g0.M * (double)g0.N * g0.K * g0.batch;
    g_zprof.flops += f;
    if (tc) g_zprof.flops_tc += f;
    return rc;
}

static int zgemm_dispatch(const Zgemm& g0, cudaStream_t s) {
    Zgemm g = g0;
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return RSRR_OK;
    if (g.K <= 0) {
        dim3 grid((unsigned)ceil_div((int64_t)g.M * g.N, 256), g.batch);
        { scale_kernel<<<grid, 256, 0, s>>>(g.C, g.M, g.N, g.ldc, g.sC, g.beta); note_launch(); }
        RSRR_CUDA(cudaGetLastError());
        return RSRR_OK;
    }
    if (g_zpath == 2 || (g_zpath == 0 && !g.fp64 && zgemm_tc_fits(g))) return zgemm_tc(g, s);
    return g.N <= 8 ? zgemm_fp64<64, 4>(g, s) : zgemm_fp64<16, 16>(g, s);
}

// ---------------------------------------------------------------------------------------------
// Norms
// ---------------------------------------------------------------------------------------------
namespace {
__device__ double block_sum(double v) {
    __shared__ double red[32];
    for (int off = 16; off; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
        for (int off = 16; off; off >>= 1) r += __shfl_down_sync(0xffffffffu, r, off);
    }
    return r;  // valid in thread 0
}

__global__ void colnorm_kernel(const c128* B, int mb, int64_t ld, double* out) {
    const int c = blockIdx.x;
    double s = 0.0;
    for (int i = threadIdx.x; i < mb; i += blockDim.x) s += cnorm2(B[i + (int64_t)c * ld]);
    s = block_sum(s);
    if (threadIdx.x == 0) out[c] = sqrt(s);
}

__global__ void blocknorm_kernel(const c128* A, int64_t lda, int r0, int r1, int c0, int c1, double* out) {
    const int64_t rows = r1 - r0;
    const int64_t total = rows * (c1 - c0);
    double s = 0.0;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = r0 + idx % rows, j = c0 + idx / rows;
        s += cnorm2(A[i + j * lda]);
    }
    s = block_sum(s);
    if (threadIdx.x == 0) atomicAdd(out, s);
}
}  // namespace

void column_norms(const c128* B, int mb, int k, int64_t ld, double* out, cudaStream_t s) {
    if (k > 0) { colnorm_kernel<<<k, 256, 0, s>>>(B, mb, ld, out); note_launch(); }
}

void block_norm2(const c128* A, int64_t lda, int r0, int r1, int c0, int c1, double* out, cudaStream_t s) {
    if (r1 <= r0 || c1 <= c0) return;
    const int64_t total = (int64_t)(r1 - r0) * (c1 - c0);
    const int blocks = (int)std::min<int64_t>(4 * 152, ceil_div(total, 256));
    { blocknorm_kernel<<<blocks, 256, 0, s>>>(A, lda, r0, r1, c0, c1, out); note_launch(); }
}

// ---------------------------------------------------------------------------------------------
// One-sided Jacobi.  A sweep is one cooperative kernel over the round-robin rounds, one CTA per
// column pair, each pair ordered after the two pairs of the previous round that held its columns.
// A pair is rotated when its inner product is above tol relative to the column norms and both
// columns are above an absolute floor: columns below the floor are rounding noise, and rotating
// them against anything changes no column above the floor by more than the floor itself.
//
// The squared column norms live in a small array: computed once at the start of the sweep and
// recomputed from the rotated entries by the CTA that rotates a pair, so they are always the sums
// a fresh pass over the stored columns would give.  A pair then costs one complex inner product
// (4 FP64 fused multiply-adds a row) when it is not rotated, nothing when a column is below the
// floor, and the columns it rotates are held in registers between the two passes.
// ---------------------------------------------------------------------------------------------
namespace {
__device__ __forceinline__ int rr_pos(int k, int r, int n) {  // player at seat k in round r
    return k == 0 ? 0 : ((k - 1 + r) % (n - 1)) + 1;
}

struct JacobiArgs {
    c128* B;
    int mb, kk, npad;
    c128* J;
    double tol, floor2, abs_g;
    double* nrm2;  // squared column norms of B (kk entries)
    int* ver;      // rounds each column has finished in this sweep (kk entries, zero at launch)
    int* jver;     // rounds whose rotation of J's column is done (kk entries, zero at launch)
    unsigned long long* max_off;
    int* rotations;  // [0] pairs rotated, [1] pairs whose inner product was formed
    GridBar gb;      // the barrier after the norms; its error word also records a wait that gave up
};

// Two block-wide sums; every thread gets both, summed in the same order (two CTA barriers).  The
// per-warp partials are combined by a shuffle tree in every warp (log2 of the warp count FP64
// additions a thread), not by a loop over them: FP64 issue slots are the scarce resource here.
__device__ __forceinline__ void block_sum2(double& a, double& b) {
    __shared__ double red2_[2][32];
    for (int off = 16; off; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
    }
    __syncthreads();
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { red2_[0][w] = a; red2_[1][w] = b; }
    __syncthreads();
    double s0 = lane < nw ? red2_[0][lane] : 0.0, s1 = lane < nw ? red2_[1][lane] : 0.0;
    for (int off = nw >> 1; off; off >>= 1) {  // nw is a power of two
        s0 += __shfl_xor_sync(0xffffffffu, s0, off);
        s1 += __shfl_xor_sync(0xffffffffu, s1, off);
    }
    a = __shfl_sync(0xffffffffu, s0, 0);
    b = __shfl_sync(0xffffffffu, s1, 0);
}

constexpr int kJacThreads = 256;
// Columns are read past L1: between rounds they are rewritten by CTAs on other SMs.
__device__ __forceinline__ c128 ldcg_c(const c128* p) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
    return mk<double>(v.x, v.y);
}
constexpr int kJacCache = 3;  // rows per thread kept in registers (columns up to 768 rows)

__device__ __forceinline__ void jac_norm_acc(double& acc, c128 x) { acc = fma(x.re, x.re, fma(x.im, x.im, acc)); }
// conj(x) y accumulated into (gr, gi)
__device__ __forceinline__ void jac_dot_acc(double& gr, double& gi, c128 x, c128 y) {
    gr = fma(x.re, y.re, fma(x.im, y.im, gr));
    gi = fma(x.re, y.im, fma(-x.im, y.re, gi));
}
// (x, y) <- (c x - sp y, s x + cp y): the rotation with the phase folded into the two complex
// coefficients (12 FP64 operations a row)
__device__ __forceinline__ void jac_rotate(c128& x, c128& y, double c, double s, c128 sp, c128 cp) {
    const c128 nx = mk<double>(fma(-sp.re, y.re, fma(sp.im, y.im, c * x.re)),
                               fma(-sp.re, y.im, fma(-sp.im, y.re, c * x.im)));
    const c128 ny = mk<double>(fma(cp.re, y.re, fma(-cp.im, y.im, s * x.re)),
                               fma(cp.re, y.im, fma(cp.im, y.re, s * x.im)));
    x = nx;
    y = ny;
}

// One column pair (p, q) of a round, p < q < kk; every thread of the CTA takes the same branches.
// Rotates the pair's columns of B and stores their norms; returns whether it rotated, with the
// rotation in (c, s, sp, cp) for J's columns, which the caller rotates after releasing B's.
// The rotation of the CTA's current pair (c, s, s e^{-i phi}, c e^{-i phi}): written by thread 0,
// read by every thread for B's columns and, after B's release, for J's.
__shared__ double jac_spar[6];

__device__ __forceinline__ bool jac_pair(const JacobiArgs& a, int p, int q) {
    const int tid = threadIdx.x;
    const double al = __ldcg(a.nrm2 + p), be = __ldcg(a.nrm2 + q);
    if (fmin(al, be) <= a.floor2) return false;
    c128* bp = a.B + (int64_t)p * a.mb;
    c128* bq = a.B + (int64_t)q * a.mb;
    c128 xc[kJacCache], yc[kJacCache];
    double gr = 0.0, gi = 0.0;
#pragma unroll
    for (int u = 0; u < kJacCache; ++u) {
        const int r = tid + kJacThreads * u;
        xc[u] = yc[u] = czero<double>();
        if (r < a.mb) {
            xc[u] = ldcg_c(bp + r);
            yc[u] = ldcg_c(bq + r);
            jac_dot_acc(gr, gi, xc[u], yc[u]);
        }
    }
    for (int r = tid + kJacThreads * kJacCache; r < a.mb; r += kJacThreads)
        jac_dot_acc(gr, gi, ldcg_c(bp + r), ldcg_c(bq + r));
    block_sum2(gr, gi);
    // the decision and the rotation are computed once, by thread 0, and shared
    __shared__ int s_act;
    if (tid == 0) {
        atomicAdd(a.rotations + 1, 1);
        int act = 0;
        const double g = sqrt(gr * gr + gi * gi);
        if (g > a.abs_g) {
            const double off = g / sqrt(al * be);
            atomicMax(a.max_off, (unsigned long long)__double_as_longlong(off));
            if (off > a.tol) {
                const double ig = 1.0 / g;
                const c128 ph = mk<double>(gr * ig, -gi * ig);  // e^{-i phi}, phi = arg(conj(b_p) b_q)
                const double zeta = (be - al) * (0.5 * ig);
                const double t = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                const double c = 1.0 / sqrt(1.0 + t * t), sn = c * t;
                jac_spar[0] = c;
                jac_spar[1] = sn;
                jac_spar[2] = ph.re * sn;
                jac_spar[3] = ph.im * sn;
                jac_spar[4] = ph.re * c;
                jac_spar[5] = ph.im * c;
                act = 1;
            }
        }
        s_act = act;
    }
    __syncthreads();
    if (!s_act) return false;
    // (b_p, b_q) <- (c b_p - s e^{-i phi} b_q, s b_p + c e^{-i phi} b_q)
    const double c = jac_spar[0], s = jac_spar[1];
    const c128 sp = mk<double>(jac_spar[2], jac_spar[3]), cp = mk<double>(jac_spar[4], jac_spar[5]);
    double an = 0.0, bn = 0.0;
#pragma unroll
    for (int u = 0; u < kJacCache; ++u) {
        const int r = tid + kJacThreads * u;
        if (r < a.mb) {
            jac_rotate(xc[u], yc[u], c, s, sp, cp);
            bp[r] = xc[u];
            bq[r] = yc[u];
            jac_norm_acc(an, xc[u]);
            jac_norm_acc(bn, yc[u]);
        }
    }
    for (int r = tid + kJacThreads * kJacCache; r < a.mb; r += kJacThreads) {
        c128 x = ldcg_c(bp + r), y = ldcg_c(bq + r);
        jac_rotate(x, y, c, s, sp, cp);
        bp[r] = x;
        bq[r] = y;
        jac_norm_acc(an, x);
        jac_norm_acc(bn, y);
    }
    block_sum2(an, bn);
    if (tid == 0) {
        a.nrm2[p] = an;
        a.nrm2[q] = bn;
        atomicAdd(a.rotations, 1);
    }
    return true;
}

// Thread 0 waits until column c has finished `target` rounds.  Bounded: after the spin limit, or
// once another CTA has reported a timeout, it records the failure and returns false.
__device__ __forceinline__ bool jac_wait(const int* ver, int c, int target, int* err) {
    const volatile int* v = ver + c;
    long long spins = 0;
    unsigned backoff = 16;
    while (*v < target) {
        if (++spins > (1LL << 24) || *(volatile int*)err != 0) {
            atomicExch(err, 1);
            return false;
        }
        __nanosleep(backoff);
        if (backoff < 256) backoff <<= 1;
    }
    return true;
}

__global__ void __launch_bounds__(kJacThreads, 3) jacobi_sweep_kernel(JacobiArgs a) {
    // One CTA per column pair (CTAs take the pairs in order, see below), so every round spreads its
    // FP64 work over all SMs.  The rounds are not separated by grid barriers: a pair of round r
    // starts as soon as both of its columns have come out of round r - 1 (a per-column count of
    // finished rounds), so a slow pair holds up only the pairs that need its columns.  The pairs,
    // their order and every value are those of the barrier-separated sweep.
    const int tid = threadIdx.x;
    __shared__ int s_ok;
    for (int c = blockIdx.x; c < a.kk; c += gridDim.x) {
        const c128* bc = a.B + (int64_t)c * a.mb;
        double s = 0.0, unused = 0.0;
        for (int r = tid; r < a.mb; r += kJacThreads) jac_norm_acc(s, ldcg_c(bc + r));
        block_sum2(s, unused);
        if (tid == 0) a.nrm2[c] = s;
    }
    if (!grid_sync(a.gb)) return;
    // The pairs of all rounds are numbered g = round * (npad / 2) + i and dealt out in that order.
    // A pair releases its columns of B (and their norms) to the next round as soon as they are
    // rotated; it then rotates its columns of J, once the previous round's rotation of them is done
    // (jver), and releases those.  With more CTAs than pairs in a round, CTAs start pairs of the next
    // round while J's rotations of this one run.  Every wait is on a smaller g (or the same g's B
    // part), every CTA takes its pairs in increasing g and all are resident (cooperative launch), so
    // the smallest unfinished step can always proceed.  The arithmetic is that of the sweep with a
    // grid barrier between rounds.
    const int ppr = a.npad / 2;
    const int64_t npairs = (int64_t)(a.npad - 1) * ppr;
    for (int64_t gi = blockIdx.x; gi < npairs; gi += gridDim.x) {
        const int round = (int)(gi / ppr), i = (int)(gi % ppr);
        int p = rr_pos(i, round, a.npad), q = rr_pos(a.npad - 1 - i, round, a.npad);
        if (p > q) { const int t = p; p = q; q = t; }
        const bool real_pair = q < a.kk;  // q == kk is the padding column of an odd count
        if (tid == 0) {
            const bool ok = jac_wait(a.ver, p, round, a.gb.err) && (!real_pair || jac_wait(a.ver, q, round, a.gb.err));
            __threadfence();
            s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) return;
        const bool rot = real_pair && jac_pair(a, p, q);
        __syncthreads();  // every store of B and of the norms issued
        if (tid == 0) {
            __threadfence();
            atomicExch(a.ver + p, round + 1);
            if (real_pair) atomicExch(a.ver + q, round + 1);
        }
        if (a.J) {
            if (tid == 0) {
                const bool ok = jac_wait(a.jver, p, round, a.gb.err) &&
                                (!real_pair || jac_wait(a.jver, q, round, a.gb.err));
                __threadfence();
                s_ok = ok;
            }
            __syncthreads();
            if (!s_ok) return;
            if (rot) {
                const double c = jac_spar[0], sn = jac_spar[1];
                const c128 sp = mk<double>(jac_spar[2], jac_spar[3]), cp = mk<double>(jac_spar[4], jac_spar[5]);
                c128* jp = a.J + (int64_t)p * a.kk;
                c128* jq = a.J + (int64_t)q * a.kk;
                for (int r = tid; r < a.kk; r += kJacThreads) {
                    c128 x = ldcg_c(jp + r), y = ldcg_c(jq + r);
                    jac_rotate(x, y, c, sn, sp, cp);
                    jp[r] = x;
                    jq[r] = y;
                }
            }
            __syncthreads();  // every store of J issued
            if (tid == 0) {
                __threadfence();
                atomicExch(a.jver + p, round + 1);
                if (real_pair) atomicExch(a.jver + q, round + 1);
            }
        }
    }
}
}  // namespace

namespace {
// out[:, i] = in[:, perm[i]] for the k columns of an m-row matrix (leading dimension m).
__global__ void gather_cols_kernel(const c128* __restrict__ in, int m, int k, const int* __restrict__ perm,
                                   c128* __restrict__ out) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)m * k) return;
    const int64_t r = idx % m, c = idx / m;
    out[idx] = in[r + (int64_t)perm[c] * m];
}
}  // namespace

int jacobi_orthogonalize(c128* B, int mb, int k, c128* J, cudaStream_t s, int max_sweeps, int* sweeps_out,
                         double abs_floor, double conv, double abs_inner) {
    if (sweeps_out) *sweeps_out = 0;
    if (k < 2) return RSRR_OK;
    const int npad = k + (k & 1);
    int dev = 0, nsm = 0, occ = 0;
    RSRR_CUDA(cudaGetDevice(&dev));
    RSRR_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    RSRR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, jacobi_sweep_kernel, kJacThreads, 0));
    if (occ < 1) return set_error(RSRR_ECUDA, "jacobi kernel cannot be resident");
    // as many CTAs as are resident (up to 4 per SM), also when that is more than a round's npad / 2
    // pairs: the surplus starts the next round's pairs while this round's J rotations finish
    const int G = (int)std::min<int64_t>((int64_t)nsm * std::min(occ, 4), (int64_t)(npad - 1) * (npad / 2));
    unsigned long long* dmax = nullptr;
    int* drot = nullptr;
    unsigned* bar = nullptr;
    double* dn2 = nullptr;
    int* dver = nullptr;
    int* djver = nullptr;
    double* dnrm = nullptr;
    int* dperm = nullptr;
    c128* tmp = nullptr;
    auto cleanup = [&]() {
        dfree(dn2, s);
        dfree(dver, s);
        dfree(djver, s);
        dfree(dmax, s);
        dfree(drot, s);
        dfree(bar, s);
        dfree(dnrm, s);
        dfree(dperm, s);
        dfree(tmp, s);
    };
    int rc = RSRR_OK;
#define JTRY(expr) do { rc = (expr); if (rc != RSRR_OK) { cleanup(); return rc; } } while (0)
    JTRY(dalloc_n(&dn2, (size_t)k, s));
    JTRY(dalloc_n(&dver, (size_t)k, s));
    JTRY(dalloc_n(&djver, (size_t)k, s));
    JTRY(dalloc_n(&dmax, 1, s));
    JTRY(dalloc_n(&drot, 2, s));
    JTRY(dalloc_n(&bar, kGridBarWords, s));
    // Before each sweep the columns (and J's with them) are put in order of decreasing norm: the
    // round-robin pairs then meet in an order that converges in fewer sweeps, and the caller,
    // which sorts the final column norms itself, sees no difference.
    JTRY(dalloc_n(&dnrm, (size_t)k, s));
    JTRY(dalloc_n(&dperm, (size_t)k, s));
    JTRY(dalloc_n(&tmp, (size_t)mb * k + (J ? (size_t)k * k : 0), s));
    if (cudaMemsetAsync(bar, 0, kGridBarWords * sizeof(unsigned), s) != cudaSuccess)
        JTRY(set_error(RSRR_ECUDA, "jacobi: clearing the grid barrier"));
#undef JTRY
    JacobiArgs ja{B, mb, k, npad, J, sqrt((double)mb) * 1.1102230246251565e-16, abs_floor * abs_floor, abs_inner,
                  dn2, dver, djver, dmax, drot, grid_bar_at(bar)};
    std::vector<double> hn(k);
    std::vector<int> order(k);
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        column_norms(B, mb, k, mb, dnrm, s);
        if (cudaMemcpyAsync(hn.data(), dnrm, (size_t)k * 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) { rc = set_error(RSRR_ECUDA, "jacobi norms"); break; }
        for (int i = 0; i < k; ++i) order[i] = i;
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return hn[a] > hn[b]; });
        bool sorted = true;
        for (int i = 0; i < k && sorted; ++i) sorted = order[i] == i;
        if (!sorted) {
            if (cudaMemcpyAsync(dperm, order.data(), (size_t)k * 4, cudaMemcpyHostToDevice, s) != cudaSuccess) {
                rc = set_error(RSRR_ECUDA, "jacobi: column order upload");
                break;
            }
            { gather_cols_kernel<<<(unsigned)ceil_div((int64_t)mb * k, 256), 256, 0, s>>>(B, mb, k, dperm, tmp); note_launch(); }
            cudaError_t ce = cudaMemcpyAsync(B, tmp, (size_t)mb * k * sizeof(c128), cudaMemcpyDeviceToDevice, s);
            if (J && ce == cudaSuccess) {
                c128* tj = tmp + (size_t)mb * k;
                { gather_cols_kernel<<<(unsigned)ceil_div((int64_t)k * k, 256), 256, 0, s>>>(J, k, k, dperm, tj); note_launch(); }
                ce = cudaMemcpyAsync(J, tj, (size_t)k * k * sizeof(c128), cudaMemcpyDeviceToDevice, s);
            }
            if (ce != cudaSuccess) { rc = set_error(RSRR_ECUDA, "jacobi: column reorder"); break; }
        }
        if (cudaMemsetAsync(dmax, 0, 8, s) != cudaSuccess || cudaMemsetAsync(drot, 0, 8, s) != cudaSuccess ||
            cudaMemsetAsync(dver, 0, (size_t)k * sizeof(int), s) != cudaSuccess ||
            cudaMemsetAsync(djver, 0, (size_t)k * sizeof(int), s) != cudaSuccess) {
            rc = set_error(RSRR_ECUDA, "jacobi: clearing the sweep counters");
            break;
        }
        void* args[] = {&ja};
        cudaEvent_t ea = nullptr, eb = nullptr;
        if (g_jprof.on) {
            cudaEventCreate(&ea);
            cudaEventCreate(&eb);
            cudaEventRecord(ea, s);
        }
        cudaError_t e = cudaLaunchCooperativeKernel((void*)jacobi_sweep_kernel, G, kJacThreads, args, 0, s);
        note_launch();
        if (g_jprof.on) {
            cudaEventRecord(eb, s);
            g_jprof.ev.emplace_back(ea, eb);
        }
        if (e != cudaSuccess) { rc = set_error(RSRR_ECUDA, cudaGetErrorString(e)); break; }
        int hrot[2] = {0, 0}, herr = 0;
        unsigned long long hmax = 0;
        if (cudaMemcpyAsync(hrot, drot, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(&herr, bar + kGridBarErrWord, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(&hmax, dmax, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) { rc = set_error(RSRR_ECUDA, "jacobi sync"); break; }
        if (herr) { rc = set_error(RSRR_ETIMEOUT, "a wait in the Jacobi sweep gave up"); break; }
        // the sweep's work: the column norms (4 real flops a row), one complex inner product for
        // every pair formed (8 a row), and for every rotated pair the rotation of both columns of
        // B and J (24 a row each) and the two new norms (8 a row)
        if (g_jprof.on)
            g_jprof.flops += 4.0 * mb * k + 8.0 * mb * hrot[1] + hrot[0] * (32.0 * mb + (J ? 24.0 * k : 0.0));
        double off;
        std::memcpy(&off, &hmax, 8);
        // converged: no rotation left, or every pair above the floor orthogonal to `conv` (the
        // remaining effect on the singular values is of second order in that number)
        if (hrot[0] == 0 || off <= conv) { ++sweep; break; }
    }
    cleanup();
    if (sweeps_out) *sweeps_out = sweep;
    return rc;
}

}  // namespace rsrr
