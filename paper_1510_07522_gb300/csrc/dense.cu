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
// memory in a fixed order (no atomics, the same bits on every run).  A product of few tiles and long K
// (32 x 8 x 100000) gives a tile several clusters, whose sums meet in a workspace (zgemm_fold_kernel).  The
// FP64 products of one pass (projection and reduced solve), before with 32 x 32 tiles of two warps
// and no K split below 512, and now: n = 9991, k_S = 133: 18.8 -> 5.0 ms (with the inverses' W, which joined
// them since); n = 900, moment scheme, k_S = 45: 18.5 -> 1.4 ms; n = 5000, k_S = 48, K = 8: 29.7 -> 3.5 ms.
// A tile is 16 x 16, or 32 x 8 and 64 x 4 (8 x 32, 4 x 64) for the products with a handful of columns (rows).
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
    int M, N, K, tm, tn, split, outer, kper;
    c128 alpha, beta;
    c128* ws;  // outer > 1: [outer][batch][N][M] sums of the clusters' K ranges
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
    constexpr int NA = (BM * BK + kZgThreads - 1) / kZgThreads, NB = (BN * BK + kZgThreads - 1) / kZgThreads;
    __shared__ c128 As[BK][BM + 1];
    __shared__ c128 Bs[BK][BN + 1];
    __shared__ c128 part[kZgTile];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    // the CTAs of a cluster are neighbouring K slices of one tile
    const int64_t cl = blockIdx.x / g.split, tile = cl / g.outer;
    const int ks = (int)(blockIdx.x % g.split), o = (int)(cl % g.outer);
    const int bm = (int)(tile % g.tm) * BM, bn = (int)((tile / g.tm) % g.tn) * BN;
    const int64_t b = tile / ((int64_t)g.tm * g.tn);
    const c128* Ab = g.A.p + b * g.A.sb;
    const c128* Bb = g.B.p + b * g.B.sb;
    const int k_begin = (int)min((int64_t)g.K, ((int64_t)o * g.split + ks) * g.kper), k_end = min(g.K, k_begin + g.kper);
    // consecutive threads follow whichever index is contiguous in memory
    const bool a_rows = g.A.sr == 1, b_rows = g.B.sr == 1;
    c128 ra[NA], rb[NB];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const int idx = tid + kZgThreads * u;
            if (idx < BM * BK) {
                const int i = a_rows ? idx % BM : idx / BK, k = a_rows ? idx / BM : idx % BK;
                ra[u] = zg_fetch(g.A, Ab, bm + i, g.M, k0 + k, k_end);
            }
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
            if (idx < BM * BK) {
                const int i = a_rows ? idx % BM : idx / BK, k = a_rows ? idx / BM : idx % BK;
                As[k][i] = ra[u];
            }
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
        if (g.outer > 1) {
            const int64_t batch = gridDim.x / ((int64_t)g.tm * g.tn * g.outer * g.split);
            g.ws[((o * batch + b) * g.N + gj) * g.M + gi] = v;
            return;
        }
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

// C = alpha sum_o ws[o] + beta C
__global__ void zgemm_fold_kernel(ZgArgs g, int64_t per_batch, int64_t total) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    c128 v = czero<double>();
    for (int o = 0; o < g.outer; ++o) v = v + g.ws[o * total + idx];
    const int64_t e = idx % per_batch;
    c128* c = g.C + idx / per_batch * g.sC + e % g.M + e / g.M * g.ldc;
    v = g.alpha * v;
    *c = (g.beta.re == 0.0 && g.beta.im == 0.0) ? v : v + g.beta * (*c);
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
    // K slices until every SM has two CTAs, but none shorter than one stage.  A cluster's eight slices are
    // followed by a second level, which costs a launch and a pass over the sums: slices of 64 terms (17 us)
    // at least to fill the SMs, of 512 to level their last wave (8 CTAs an SM).
    const int64_t tiles = (int64_t)a.tm * a.tn * g.batch, nsm = sm_count();
    int split = 1;
    while (split < kZgMaxSplit && tiles * split < 2 * nsm && g.K >= 2 * split * BK) split *= 2;
    auto clusters = [&](int64_t ctas, int64_t terms) { return std::min(ctas / (tiles * split), g.K / (split * terms)); };
    const int64_t outer = split < kZgMaxSplit ? 1 : std::max({(int64_t)1, clusters(2 * nsm, 64), clusters(8 * nsm, 512)});
    a.split = split;
    a.outer = (int)outer;
    a.kper = (int)ceil_div(g.K, split * outer);
    if (tiles * split * outer > INT32_MAX) return set_error(RSRR_EINVAL, "zgemm: too many tiles");
    const int64_t per_batch = (int64_t)g.M * g.N, total = per_batch * g.batch;
    a.ws = nullptr;
    if (outer > 1) RSRR_TRY(dalloc_n(&a.ws, (size_t)(outer * total), s));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * split * outer));
    cfg.blockDim = dim3(kZgThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = split;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, zgemm_kernel<BM, BN>, a);
    note_launch();
    if (outer > 1) {
        if (e == cudaSuccess) {
            { zgemm_fold_kernel<<<(unsigned)ceil_div(total, 256), 256, 0, s>>>(a, per_batch, total); note_launch(); }
            e = cudaGetLastError();
        }
        dfree(a.ws, s);
    }
    return e == cudaSuccess ? RSRR_OK : set_error(RSRR_ECUDA, std::string("zgemm: ") + cudaGetErrorString(e));
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
    const bool tc = !g0.fp64 && (g_zpath == 2 || (g_zpath == 0 && zgemm_tc_fits(g0)));
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
    if (!g.fp64 && (g_zpath == 2 || (g_zpath == 0 && zgemm_tc_fits(g)))) return zgemm_tc(g, s);
    if (g.N <= 4) return zgemm_fp64<64, 4>(g, s);
    if (g.N <= 8) return zgemm_fp64<32, 8>(g, s);
    if (g.M <= 4) return zgemm_fp64<4, 64>(g, s);
    return g.M <= 8 ? zgemm_fp64<8, 32>(g, s) : zgemm_fp64<16, 16>(g, s);
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
    const int blocks = (int)std::min<int64_t>(4 * sm_count(), ceil_div(total, 256));
    { blocknorm_kernel<<<blocks, 256, 0, s>>>(A, lda, r0, r1, c0, c1, out); note_launch(); }
}

// ---------------------------------------------------------------------------------------------
// One-sided Jacobi.  A sweep is one cooperative kernel over the round-robin rounds, one CTA per
// column pair, each pair ordered after the two pairs of the previous round that held its columns.
// A pair is rotated when its inner product is above tol relative to the column norms and both
// columns are above an absolute floor: columns below the floor are rounding noise, and rotating
// them against anything changes no column above the floor by more than the floor itself.
//
// The rounds of a sweep are a chain, so a pair's latency is what counts, and on this part a
// dependent FP64 operation takes 70-85 ns, a division 260 ns, a square root 350 ns.  A pair is
// therefore one pass: both columns are loaded into registers with the first reads, one reduction
// gives the inner product and both norms, and the rotation comes from two FP64 reciprocal square
// roots (an FP32 seed and one third-order step each, four dependent operations).  With the angle in
// FP32 a whole pass took 0.3 to 1.2 % less (70.2 instead of 70.7 ms at n = 900), but a pair kept 2^-23 of its
// inner product and two columns needed a third sweep.
// One round took 3.0 us at 212 columns, from 6.1 us (with the angle still in FP32); a whole pass's sweeps: n = 900,
// k_S = 233: 50.7 -> 18.7 ms, n = 40000: 88.9 -> 43.5 ms (there also without J in the projection, see project.cu), and
// with the rounds over the columns above the floor only, in FP64: 11.9 and 20.9 ms.
// The norms that decide about the floor are al - Re(conj(T) g) and be + Re(conj(T) g), T the rotation's
// complex tangent: to rounding in the larger one (of two nearly parallel columns the smaller one keeps few digits;
// such a pair is rotated, so another sweep follows with fresh norms).  Every pair forms its own from the columns.
// ---------------------------------------------------------------------------------------------
namespace {
__device__ __forceinline__ int rr_pos(int k, int r, int n) {  // player at seat k in round r
    return k == 0 ? 0 : ((k - 1 + r) % (n - 1)) + 1;
}

struct JacobiCtl {  // cleared before each sweep
    unsigned long long max_off;
    int rotations, formed;  // pairs rotated, pairs whose inner product was formed
    int err, pad[3];
};
struct JacobiArgs {
    c128* B;
    int mb, kk, npad;  // rows of B; columns of the round robin, rounded up to even in npad
    c128* J;
    int ldj;           // rows of J
    double tol2, floor2;
    double* nrm2;    // squared column norms of B
    // rounds each column has finished in this sweep, rounds whose rotation of J's column is done (zero
    // at launch); one entry every kJacVer words, so that the polls of a round spread over L2
    unsigned *ver, *jver;
    JacobiCtl* ctl;
};

// Columns are read past L1: between rounds they are rewritten by CTAs on other SMs.
__device__ __forceinline__ c128 ldcg_c(const c128* p) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
    return mk<double>(v.x, v.y);
}
constexpr int kJacCache = 3;  // rows per thread kept in registers
constexpr int kJacVer = 8;

// x^(-1/2) to FP64 rounding for x in FP32's normal range
__device__ __forceinline__ double rsqrt_mid(double x) {
    const double y = (double)rsqrtf((float)x), r = fma(-(x * y), y, 1.0);
    return fma(fma(0.375, r, 0.5), y * r, y);
}

struct JacSums { double gr, gi, al, be; };
__device__ __forceinline__ void jac_acc(JacSums& t, c128 x, c128 y) {
    t.gr = fma(x.re, y.re, fma(x.im, y.im, t.gr));  // conj(x) y
    t.gi = fma(x.re, y.im, fma(-x.im, y.re, t.gi));
    t.al = fma(x.re, x.re, fma(x.im, x.im, t.al));
    t.be = fma(y.re, y.re, fma(y.im, y.im, t.be));
}
// (x, y) <- (c x - conj(S) y, S x + c y): 12 FP64 operations a row
__device__ __forceinline__ void jac_rotate(c128& x, c128& y, double c, c128 S) {
    const c128 nx = mk<double>(fma(-S.re, y.re, fma(-S.im, y.im, c * x.re)),
                               fma(-S.re, y.im, fma(S.im, y.re, c * x.im)));
    const c128 ny = mk<double>(fma(S.re, x.re, fma(-S.im, x.im, c * y.re)),
                               fma(S.re, x.im, fma(S.im, x.re, c * y.im)));
    x = nx;
    y = ny;
}

// The sums of the four values over the CTA, in every lane of warp 0 (lane l holds value l & 3).  A
// full-warp FP64 addition takes 64 clocks of its sub-partition, so the values are reduce-scattered.
template <int NT>
__device__ __forceinline__ double jac_reduce(JacSums t) {
    constexpr int NW = NT / 32;
    __shared__ double red[NW * 4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool h1 = lane & 1, h2 = lane & 2;
    double a = (h1 ? t.gi : t.gr) + __shfl_xor_sync(0xffffffffu, h1 ? t.gr : t.gi, 1);
    double b = (h1 ? t.be : t.al) + __shfl_xor_sync(0xffffffffu, h1 ? t.al : t.be, 1);
    double v = (h2 ? b : a) + __shfl_xor_sync(0xffffffffu, h2 ? a : b, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    if (lane < 4) red[warp * 4 + lane] = v;
    __syncthreads();
    if (warp == 0) {
        v = red[lane % (NW * 4)];
        for (int off = 4; off < 4 * NW; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    }
    return v;
}

// Waits until column c has finished `target` rounds.  Bounded: after the spin limit, or once
// another CTA has reported a timeout, it records the failure and returns false.
__device__ __forceinline__ bool jac_wait(const unsigned* ver, int c, unsigned target, int* err) {
    long long spins = 0;
    while (ld_acquire_gpu(ver + (int64_t)c * kJacVer) < target) {
        if (++spins > (1LL << 22) || ((spins & 255) == 0 && *(volatile int*)err != 0)) {
            atomicExch(err, 1);
            return false;
        }
    }
    return true;
}

template <int NT>
__global__ void __launch_bounds__(NT, 768 / NT) jacobi_sweep_kernel(JacobiArgs a) {
    // One CTA per column pair, so every round spreads its FP64 work over all SMs.  The rounds are not
    // separated by grid barriers: a pair of round r starts as soon as both of its columns have come out
    // of round r - 1 (a per-column count of finished rounds), so a slow pair holds up only the pairs
    // that need its columns.  The pairs of all rounds are numbered g = round * (npad / 2) + i and
    // dealt out in that order.  A pair releases its columns of B to the next round as soon as they are
    // rotated; it then rotates its columns of J, once the previous round's rotation of them is done
    // (jver), and releases those.  With more CTAs than pairs in a round, CTAs start pairs of the next
    // round meanwhile.  Every wait is on a smaller g (or the same g's B part), every CTA takes its pairs
    // in increasing g and all are resident (cooperative launch), so the smallest unfinished step can
    // always proceed.
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ int s_ok, s_act;
    __shared__ double s_c;
    __shared__ c128 s_S;
    const int ppr = a.npad / 2;
    const int64_t npairs = (int64_t)(a.npad - 1) * ppr;
    for (int64_t g = blockIdx.x; g < npairs; g += gridDim.x) {
        const unsigned round = (unsigned)(g / ppr);
        const int i = (int)(g % ppr);
        int p = rr_pos(i, (int)round, a.npad), q = rr_pos(a.npad - 1 - i, (int)round, a.npad);
        if (p > q) { const int t = p; p = q; q = t; }
        const bool real_pair = q < a.kk;  // q == kk is the padding column of an odd count
        auto wait_both = [&](const unsigned* ver) {  // lanes 0 and 1 of warp 0 poll one column each
            if (warp == 0) {
                bool ok = true;
                if (lane < (real_pair ? 2 : 1)) ok = jac_wait(ver, lane ? q : p, round, &a.ctl->err);
                ok = __all_sync(0xffffffffu, ok);
                if (lane == 0) s_ok = ok;
            }
            __syncthreads();
            return s_ok != 0;
        };
        auto release_both = [&](unsigned* ver) {  // after a barrier: every store of the columns is issued
            if (tid < (real_pair ? 2 : 1)) st_release_gpu(ver + (int64_t)(tid ? q : p) * kJacVer, round + 1);
        };
        if (!wait_both(a.ver)) return;
        bool rot = false;
        if (real_pair) {
            c128* bp = a.B + (int64_t)p * a.mb;
            c128* bq = a.B + (int64_t)q * a.mb;
            const double np = __ldcg(a.nrm2 + p), nq = __ldcg(a.nrm2 + q);
            c128 xc[kJacCache], yc[kJacCache];
#pragma unroll
            for (int u = 0; u < kJacCache; ++u) {
                const int r = tid + NT * u;
                xc[u] = yc[u] = czero<double>();
                if (r < a.mb) {
                    xc[u] = ldcg_c(bp + r);
                    yc[u] = ldcg_c(bq + r);
                }
            }
            if (fmin(np, nq) > a.floor2) {  // the same for the whole CTA
                JacSums t{0.0, 0.0, 0.0, 0.0};
#pragma unroll
                for (int u = 0; u < kJacCache; ++u)
                    if (tid + NT * u < a.mb) jac_acc(t, xc[u], yc[u]);
                for (int r = tid + NT * kJacCache; r < a.mb; r += NT) jac_acc(t, ldcg_c(bp + r), ldcg_c(bq + r));
                const double v = jac_reduce<NT>(t);
                if (warp == 0) {
                    const double gr = __shfl_sync(0xffffffffu, v, 0), gi = __shfl_sync(0xffffffffu, v, 1);
                    const double al = __shfl_sync(0xffffffffu, v, 2), be = __shfl_sync(0xffffffffu, v, 3);
                    const double g2 = fma(gr, gr, gi * gi), ab = al * be;
                    const bool act = g2 > 0.0 && g2 > a.tol2 * ab;
                    double dn = 0.0;
                    if (act) {
                        // With d = be - al and h = sqrt(d^2 + 4 |g|^2): cos 2 theta = |d| / h, sin 2 theta = 2 |g| / h, so
                        // c^2 = (1 + |d| / h) / 2 and S = s e^{i phi} = g sign(d) / (h c); d and g are scaled by a power of two
                        const int e = max(1, min(2045, (__double2hiint(fmax(al, be)) >> 20) & 0x7ff));
                        const double sf = __hiloint2double((2046 - e) << 20, 0);
                        const double fr = gr * sf, fi = gi * sf, d = (be - al) * sf;
                        const double ih = rsqrt_mid(fma(d, d, 4.0 * fma(fr, fr, fi * fi)));
                        const double c2 = fma(0.5 * fabs(d), ih, 0.5), ic = rsqrt_mid(c2);
                        const double w = copysign(ih * ic, d);
                        const c128 S = mk<double>(fr * w, fi * w);
                        dn = fma(S.re, gr, S.im * gi) * ic;  // Re(conj(T) g), T = S / c
                        if (lane == 0) {
                            s_c = c2 * ic;
                            s_S = S;
                        }
                    }
                    if (lane == 0) {
                        s_act = act;
                        atomicAdd(&a.ctl->formed, 1);
                        if (act) {
                            a.nrm2[p] = al - dn;
                            a.nrm2[q] = be + dn;
                            atomicAdd(&a.ctl->rotations, 1);
                        }
                    } else if (lane == 1 && g2 > 0.0) {
                        atomicMax(&a.ctl->max_off, (unsigned long long)__double_as_longlong(sqrt(g2 / ab)));
                    }
                }
                __syncthreads();
                rot = s_act != 0;
                if (rot) {
                    const double c = s_c;
                    const c128 S = s_S;
#pragma unroll
                    for (int u = 0; u < kJacCache; ++u) {
                        const int r = tid + NT * u;
                        if (r < a.mb) {
                            jac_rotate(xc[u], yc[u], c, S);
                            bp[r] = xc[u];
                            bq[r] = yc[u];
                        }
                    }
                    for (int r = tid + NT * kJacCache; r < a.mb; r += NT) {
                        c128 x = ldcg_c(bp + r), y = ldcg_c(bq + r);
                        jac_rotate(x, y, c, S);
                        bp[r] = x;
                        bq[r] = y;
                    }
                }
            }
        }
        __syncthreads();
        release_both(a.ver);
        if (a.J) {
            if (!wait_both(a.jver)) return;
            if (rot) {
                const double c = s_c;
                const c128 S = s_S;
                c128* jp = a.J + (int64_t)p * a.ldj;
                c128* jq = a.J + (int64_t)q * a.ldj;
                for (int r = tid; r < a.ldj; r += NT) {
                    c128 x = ldcg_c(jp + r), y = ldcg_c(jq + r);
                    jac_rotate(x, y, c, S);
                    jp[r] = x;
                    jq[r] = y;
                }
            }
            __syncthreads();
            release_both(a.jver);
        }
    }
}

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
                         double abs_floor, double conv) {
    if (sweeps_out) *sweeps_out = 0;
    if (k < 2) return RSRR_OK;
    // 128 threads while they hold the columns in registers: fewer warps to sum over
    const bool small = mb <= 128 * kJacCache;
    const void* kern = small ? (const void*)jacobi_sweep_kernel<128> : (const void*)jacobi_sweep_kernel<256>;
    const int threads = small ? 128 : 256;
    int dev = 0, nsm = 0, occ = 0;
    RSRR_CUDA(cudaGetDevice(&dev));
    RSRR_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    RSRR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, 0));
    if (occ < 1) return set_error(RSRR_ECUDA, "jacobi kernel cannot be resident");
    // One CTA a pair where all are resident.  With J, twice as many: the surplus starts the next
    // round's pairs while this round's J rotations finish.  More would only poll: with four CTAs an
    // SM and the counts packed in a few lines a round took 5.7 us instead of 3.0.
    const int max_ctas = nsm * std::min(occ, 4);
    const size_t ctl_bytes = sizeof(JacobiCtl) + (size_t)2 * k * kJacVer * sizeof(unsigned);
    const size_t ord_bytes = (size_t)k * (sizeof(double) + sizeof(int));  // squared norms, then the order
    uint8_t *ctl = nullptr, *ord = nullptr;
    double* dnrm = nullptr;
    c128* tmp = nullptr;
    auto cleanup = [&]() {
        for (void* p : {(void*)ctl, (void*)ord, (void*)dnrm, (void*)tmp}) dfree(p, s);
    };
    int rc = RSRR_OK;
#define JTRY(expr) do { rc = (expr); if (rc != RSRR_OK) { cleanup(); return rc; } } while (0)
    JTRY(dalloc_n(&ctl, ctl_bytes, s));
    JTRY(dalloc_n(&ord, ord_bytes, s));
    // Before each sweep the columns (and J's with them) are put in order of decreasing norm: the
    // round-robin pairs then meet in an order that converges in fewer sweeps, and the caller,
    // which sorts the final column norms itself, sees no difference.
    JTRY(dalloc_n(&dnrm, (size_t)k, s));
    JTRY(dalloc_n(&tmp, (size_t)mb * k + (J ? (size_t)k * k : 0), s));
#undef JTRY
    c128 *curB = B, *altB = tmp, *curJ = J, *altJ = J ? tmp + (size_t)mb * k : nullptr;
    JacobiCtl* dctl = reinterpret_cast<JacobiCtl*>(ctl);
    JacobiArgs ja{};
    ja.mb = mb;
    ja.ldj = k;
    ja.tol2 = (double)mb * 1.1102230246251565e-16 * 1.1102230246251565e-16;
    ja.floor2 = abs_floor * abs_floor;
    ja.nrm2 = reinterpret_cast<double*>(ord);
    ja.ver = reinterpret_cast<unsigned*>(ctl + sizeof(JacobiCtl));
    ja.jver = ja.ver + (size_t)k * kJacVer;
    ja.ctl = dctl;
    int* dperm = reinterpret_cast<int*>(ord + (size_t)k * sizeof(double));
    std::vector<double> hn(k);
    std::vector<int> order(k);
    std::vector<uint8_t> hord(ord_bytes);
    int sweep = 0;
    auto fetch_norms = [&]() {  // queued; the next sweep sorts by them
        column_norms(curB, mb, k, mb, dnrm, s);
        return cudaMemcpyAsync(hn.data(), dnrm, (size_t)k * 8, cudaMemcpyDeviceToHost, s) == cudaSuccess;
    };
    if (!fetch_norms() || cudaStreamSynchronize(s) != cudaSuccess) rc = set_error(RSRR_ECUDA, "jacobi norms");
    for (; rc == RSRR_OK && sweep < max_sweeps; ++sweep) {
        for (int i = 0; i < k; ++i) order[i] = i;
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return hn[a] > hn[b]; });
        bool sorted = true;
        for (int i = 0; i < k; ++i) {
            sorted = sorted && order[i] == i;
            const double n2 = hn[order[i]] * hn[order[i]];
            std::memcpy(hord.data() + (size_t)i * 8, &n2, 8);
        }
        std::memcpy(hord.data() + (size_t)k * 8, order.data(), (size_t)k * 4);
        if (cudaMemcpyAsync(ord, hord.data(), ord_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaMemsetAsync(ctl, 0, ctl_bytes, s) != cudaSuccess) {
            rc = set_error(RSRR_ECUDA, "jacobi: column order and counters");
            break;
        }
        if (!sorted) {
            { gather_cols_kernel<<<(unsigned)ceil_div((int64_t)mb * k, 256), 256, 0, s>>>(curB, mb, k, dperm, altB); note_launch(); }
            std::swap(curB, altB);
            if (J) {
                { gather_cols_kernel<<<(unsigned)ceil_div((int64_t)k * k, 256), 256, 0, s>>>(curJ, k, k, dperm, altJ); note_launch(); }
                std::swap(curJ, altJ);
            }
        }
        // Only the columns above the floor can be rotated, and they come first: the round robin runs
        // over those.  (A Hankel matrix has as many as the contour encloses eigenvalues, and some:
        // 30 of 466 at n = 900, where a sweep took 0.95 ms for its 465 rounds whatever they rotated, now
        // 0.12; the sweeps of a pass at n = 40000: 43.3 -> 19.8 ms.)
        int active = 0;
        while (active < k && hn[order[active]] > abs_floor) ++active;
        if (active < 2) { ++sweep; break; }
        ja.kk = active;
        ja.npad = active + (active & 1);
        ja.B = curB;
        ja.J = curJ;
        const int G = std::min(max_ctas, (J ? 2 : 1) * (ja.npad / 2));
        void* args[] = {&ja};
        cudaEvent_t ea = nullptr, eb = nullptr;
        if (g_jprof.on) {
            cudaEventCreate(&ea);
            cudaEventCreate(&eb);
            cudaEventRecord(ea, s);
        }
        cudaError_t e = cudaLaunchCooperativeKernel(kern, G, threads, args, 0, s);
        note_launch();
        if (g_jprof.on) {
            cudaEventRecord(eb, s);
            g_jprof.ev.emplace_back(ea, eb);
        }
        if (e != cudaSuccess) { rc = set_error(RSRR_ECUDA, cudaGetErrorString(e)); break; }
        JacobiCtl hc;
        if (cudaMemcpyAsync(&hc, dctl, sizeof(hc), cudaMemcpyDeviceToHost, s) != cudaSuccess || !fetch_norms() ||
            cudaStreamSynchronize(s) != cudaSuccess) { rc = set_error(RSRR_ECUDA, "jacobi sync"); break; }
        if (hc.err) { rc = set_error(RSRR_ETIMEOUT, "a wait in the Jacobi sweep gave up"); break; }
        // the sweep's work: one complex inner product and two norms for every pair formed (16 real
        // flops a row), and for every rotated pair the rotation of both columns of B and J (24 a row)
        if (g_jprof.on) g_jprof.flops += 16.0 * mb * hc.formed + hc.rotations * (24.0 * mb + (J ? 24.0 * k : 0.0));
        double off;
        std::memcpy(&off, &hc.max_off, 8);
        // converged: no rotation left, or every pair above the floor orthogonal to `conv` (the
        // remaining effect on the singular values is of second order in that number)
        if (hc.rotations == 0 || off <= conv) { ++sweep; break; }
    }
    if (rc == RSRR_OK && curB != B &&
        (cudaMemcpyAsync(B, curB, (size_t)mb * k * sizeof(c128), cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
         (J && cudaMemcpyAsync(J, curJ, (size_t)k * k * sizeof(c128), cudaMemcpyDeviceToDevice, s) != cudaSuccess)))
        rc = set_error(RSRR_ECUDA, "jacobi: copy of the columns");
    cleanup();
    if (sweeps_out) *sweeps_out = sweep;
    return rc;
}

}  // namespace rsrr
