// Dense complex LU with partial pivoting, one thread-block cluster (1, 2, 4 or 8 CTAs) per sampling
// point, and its block solves.
//
// Factorisation of one point (right-looking, panels of NB = 64 columns):
//   1. panel: the m x 64 panel is factored as two 32-column leaves (left leaf, its
//      interchanges and L11^{-1} applied to the right half, rank-32 update of the right half,
//      right leaf, its interchanges applied back to the left half).  A leaf is column-by-
//      column getf2 (pivot by cabs1 = |re| + |im|, lowest row on ties).  Panels of at most
//      ~380 (complex64) / ~190 (complex128) rows are staged in shared memory whole, taller ones by
//      leaves of 16, 8 or 4 columns.
//   2. the panel's 64 interchanges are composed into one permutation of the <= 128 rows they
//      touch; inv(L11) and inv(U11) of the diagonal block are formed once.
//   3. trailing rows: per block of columns, the touched rows are gathered, permuted, and the
//      64 pivot rows become U12 = inv(L11) * (permuted rows)  (one small product).
//   4. trailing update A22 -= L21 * U12: 128 x 128 (complex64) or 64 x 64 (complex128) tiles,
//      L21 tiles double-buffered in shared memory by cp.async, U12 block resident, each
//      thread holding an 8 x 8 (4 x 4) block of the tile in registers.
// The update is the dense contraction that carries (8/3) n^3 real flops per point; steps 1-3
// are O(n^2 NB), but they, the operand images and the FP64 residuals took 52 of the 62 ms of a point at
// n = 1600.  With leaves in shared memory, 16-byte image stores, four columns a thread in step 3 and T
// kept for the residuals, a pass of 32 such points takes 38 ms on 32 CTAs, and 16 ms with a cluster of
// four CTAs a point (CTA 0 factors the panels, everything else is dealt out).
#include <algorithm>
#include <climits>
#include <functional>
#include <queue>
#include <string>
#include <vector>

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "dense_lu.cuh"
#include "tc.cuh"

namespace rsrr {

namespace cg = cooperative_groups;

namespace {
using namespace tc;

constexpr int NB = kDenseNB;
constexpr int NBP = NB + 1;  // padded row length of the diagonal-block arrays in shared memory
constexpr int NT = kDenseThreads;
constexpr int NW = NT / 32;
constexpr unsigned FULL = 0xffffffffu;

// Barrier of the NT worker threads (warps 0..7).  The complex64 factor kernel adds a ninth warp
// that feeds the tensor cores and never takes part in the workers' barriers.
__device__ __forceinline__ void wsync() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

template <typename R> struct DTile;
template <> struct DTile<float> { static constexpr int TM = 128, TN = 128; };  // trailing rows only
template <> struct DTile<double> { static constexpr int TM = 64, TN = 64, MI = 4, MJ = 4; };

template <typename R>
constexpr size_t gemm_smem() {
    return (2 * (size_t)NB * DTile<R>::TM + (size_t)NB * (DTile<R>::TN + 1)) * sizeof(cplx<R>);
}
template <typename R>
constexpr size_t rows_smem() {
    return ((size_t)NB * NBP + (size_t)2 * NB * DTile<R>::TN) * sizeof(cplx<R>);
}
template <typename R>
constexpr size_t inverse_smem() {
    return (size_t)3 * NB * NBP * sizeof(cplx<R>);
}
// Tensor-core trailing update (complex64): an L21 tile of 128 rows and a U12 block of 128
// columns, each as six BF16 arrays (re hi, mid, lo; im hi, mid, lo) with K = 64 (one 128-byte
// row) in the swizzled K-major layout the MMA reads; +1024 B to align the operand base.
constexpr uint32_t TC_ROWS = 128, TC_COLS = 128;
constexpr uint32_t TC_SPLIT = 3;                                     // bf16 pieces per FP32 value
constexpr uint32_t TC_ARR = 2 * TC_SPLIT;                           // arrays per operand
constexpr uint32_t TC_A_BYTES = TC_ARR * TC_ROWS * NB * 2;          // 96 KB
constexpr uint32_t TC_B_BYTES = TC_ARR * TC_COLS * NB * 2;          // 96 KB
constexpr uint32_t TC_A_FLOATS = TC_A_BYTES / 4, TC_B_FLOATS = TC_B_BYTES / 4;  // image sizes in 4-byte words
constexpr uint32_t TC_TMEM_COLS = 512;               // two accumulator buffers of (128 re + 128 im) columns
constexpr size_t tc_smem() { return (size_t)TC_A_BYTES + TC_B_BYTES + 1024; }

template <typename R>
constexpr size_t factor_smem() {
    return std::max(sizeof(R) == 4 ? tc_smem() : gemm_smem<R>(), std::max(rows_smem<R>(), inverse_smem<R>()));
}

struct DShared {
    uint64_t cbar;      // the cluster's barrier: one arrival per CTA
    int cok;
    int cabort;         // a CTA of the cluster has given up
    double2 u12[32 * 32];  // U12 of the panel's left leaf (32 x 32, complex64 or complex128)
    int piv[NB];        // panel pivots, relative to the panel's first row
    int rows[2 * NB];   // composed interchanges: row rows[e] receives row src[e]
    int src[2 * NB];
    int cnt;
    int res;
    int info;
    int job;
    int red_i[NW];
    unsigned red_u[NW];
    double red_v[NW];
};

// The worker threads of the cluster's CTAs.  `fail` is sticky and the same for all of a CTA's workers.
struct Cluster {
    int rank = 0, size = 1;
    uint32_t phase = 0;
    bool fail = false;
    unsigned long long polls = 0;  // of one wait (dense_wait_polls)
};

// The CTA gives up: the others of the cluster leave their waits too.
__device__ __forceinline__ void cluster_fail(Cluster& c, DShared& sh) {
    if (!c.fail && (int)threadIdx.x < c.size) *(volatile int*)cg::this_cluster().map_shared_rank(&sh.cabort, threadIdx.x) = 1;
    c.fail = true;
}

// Barrier of all workers of the cluster, ordering their global and shared memory accesses.  The
// hardware cluster barrier counts every thread, and the tensor-core producer warp takes no part, so the
// CTAs arrive on one another's mbarrier.  Bounded by what another CTA may do in between
// (dense_wait_polls): when a wait gives up, `fail` is set here, no later one is entered, and the other CTAs'
// waits end at once.
__device__ __forceinline__ bool csync(Cluster& c, DShared& sh) {
    wsync();
    if (c.size == 1 || c.fail) return !c.fail;
    if ((int)threadIdx.x < c.size) {
        __threadfence();
        asm volatile("{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n"
                     " mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n}\n" ::"r"(smem_u32(&sh.cbar)),
                     "r"(threadIdx.x) : "memory");
    }
    if (threadIdx.x == 0) {
        uint32_t done = 0;
        for (unsigned long long it = 0; it < c.polls && !done; ++it) {
            asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                         " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(smem_u32(&sh.cbar)), "r"(c.phase) : "memory");
            if (!done && it > 4096) {
                __nanosleep(64);
                if ((it & 63) == 0 && *(volatile int*)&sh.cabort) break;
            }
        }
        __threadfence();
        sh.cok = (int)done;
    }
    wsync();
    c.phase ^= 1;
    if (!sh.cok) cluster_fail(c, sh);
    return !c.fail;
}

template <typename R>
__device__ __forceinline__ cplx<R>* sh_u12(DShared& sh) { return reinterpret_cast<cplx<R>*>(sh.u12); }

// ------------------------------------------------------------------------------------------
// cp.async element copies (src_bytes = 0 fills zeros; the source must still be a valid address)
// ------------------------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void cp_elem(cplx<R>* smem, const cplx<R>* gmem, bool valid) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    if (sizeof(cplx<R>) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(valid ? 16 : 0));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(valid ? 8 : 0));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// Row of the largest cabs1 in col[c..m) (lowest row on ties; c if every entry is NaN).  Complex64
// compares the bit patterns (non-negative floats order like integers) with warp reductions of the
// integer pipe: a conversion to FP64 would cost 64 clocks a warp and row.
template <typename R>
__device__ int col_argmax(const cplx<R>* col, int c, int m, DShared& sh) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if constexpr (sizeof(R) == 4) {
        unsigned best = 0;  // 1 + bits of the largest value so far
        int bi = INT_MAX;
        for (int r = c + (int)threadIdx.x; r < m; r += NT) {
            const float a = cabs1(col[r]);
            const unsigned key = a >= 0.f ? __float_as_uint(a) + 1u : 0u;  // 0: NaN
            if (key > best) { best = key; bi = r; }
        }
        const unsigned top = __reduce_max_sync(FULL, best);
        const int row = (int)__reduce_min_sync(FULL, (unsigned)(best == top ? bi : INT_MAX));
        if (lane == 0) { sh.red_u[w] = top; sh.red_i[w] = row; }
        wsync();
        best = lane < NW ? sh.red_u[lane] : 0u;
        bi = lane < NW ? sh.red_i[lane] : INT_MAX;
        const unsigned all = __reduce_max_sync(FULL, best);
        const int res = (int)__reduce_min_sync(FULL, (unsigned)(best == all ? bi : INT_MAX));
        return res == INT_MAX ? c : res;
    } else {
        double best = -1.0;
        int bi = INT_MAX;
        for (int r = c + (int)threadIdx.x; r < m; r += NT) {
            const double a = (double)cabs1(col[r]);
            if (a > best) { best = a; bi = r; }
        }
        for (int off = 16; off; off >>= 1) {
            const double ob = __shfl_down_sync(FULL, best, off);
            const int oi = __shfl_down_sync(FULL, bi, off);
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (lane == 0) { sh.red_v[w] = best; sh.red_i[w] = bi; }
        wsync();
        if (w == 0) {
            best = lane < NW ? sh.red_v[lane] : -1.0;
            bi = lane < NW ? sh.red_i[lane] : INT_MAX;
            for (int off = 16; off; off >>= 1) {
                const double ob = __shfl_down_sync(FULL, best, off);
                const int oi = __shfl_down_sync(FULL, bi, off);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (lane == 0) sh.res = (bi == INT_MAX) ? c : bi;
        }
        wsync();
        return sh.res;
    }
}

// getf2 on the m x w block P (leading dimension ld): pivots piv[c] relative to row 0.
template <typename R>
__device__ void leaf_factor(cplx<R>* P, int64_t ld, int m, int w, int* piv, int col_base, DShared& sh) {
    for (int c = 0; c < w; ++c) {
        cplx<R>* colc = P + (int64_t)c * ld;
        const int p = col_argmax(colc, c, m, sh);
        if (threadIdx.x == 0) piv[c] = p;
        // the interchange, and U row c of the leaf in shared memory (read by every thread); each row's
        // entries are loaded in chunks before any is stored, so a tall leaf in global memory pays the
        // memory latency once per chunk instead of once per column.
        cplx<R>* urow = sh_u12<R>(sh);
        if ((int)threadIdx.x < w) {
            cplx<R>* cq = P + (int64_t)threadIdx.x * ld;
            const cplx<R> t = cq[p];
            urow[threadIdx.x] = t;
            if (p != c) {
                cq[p] = cq[c];
                cq[c] = t;
            }
        }
        wsync();
        const cplx<R> pv = urow[c];
        const bool zero = cis_zero(pv);
        if (zero && threadIdx.x == 0 && sh.info == 0) sh.info = col_base + c + 1;
        const cplx<R> rp = zero ? czero<R>() : crecip(pv);
        constexpr int QL = sizeof(R) == 4 ? 16 : 8;
        for (int r = c + 1 + (int)threadIdx.x; r < m; r += NT) {
            cplx<R> l = colc[r];
            if (!zero) {
                l = l * rp;
                colc[r] = l;
            }
            for (int q0 = c + 1; q0 < w; q0 += QL) {
                cplx<R> x[QL];
#pragma unroll
                for (int j = 0; j < QL; ++j)
                    x[j] = (q0 + j < w) ? P[r + (int64_t)(q0 + j) * ld] : czero<R>();
#pragma unroll
                for (int j = 0; j < QL; ++j)
                    if (q0 + j < w) {
                        cfms(x[j], l, urow[q0 + j]);
                        P[r + (int64_t)(q0 + j) * ld] = x[j];
                    }
            }
        }
        wsync();
    }
}

// Factor the m x nbk panel P as two leaves of 32 columns; sh.piv[0..nbk) relative to row 0,
// with every interchange applied to all nbk columns.
template <typename R>
__device__ void panel_factor(cplx<R>* P, int64_t ld, int m, int nbk, int col_base, DShared& sh) {
    const int w1 = min(32, nbk);
    leaf_factor(P, ld, m, w1, sh.piv, col_base, sh);
    if (nbk <= w1) return;
    const int w2 = nbk - w1;  // w1 == 32 from here on
    cplx<R>* Rt = P + (int64_t)w1 * ld;
    for (int q = threadIdx.x; q < w2; q += NT) {  // left interchanges on the right half
        cplx<R>* cq = Rt + (int64_t)q * ld;
        for (int c = 0; c < w1; ++c) {
            const int p = sh.piv[c];
            if (p != c) {
                const cplx<R> t = cq[c];
                cq[c] = cq[p];
                cq[p] = t;
            }
        }
    }
    wsync();
    for (int q = threadIdx.x; q < w2; q += NT) {  // U12 = L11^{-1} (top 32 rows of the right half)
        cplx<R>* cq = Rt + (int64_t)q * ld;
        for (int r = 1; r < w1; ++r) {
            cplx<R> acc = cq[r];
            for (int s = 0; s < r; ++s) cfms(acc, P[r + (int64_t)s * ld], cq[s]);
            cq[r] = acc;
        }
    }
    wsync();
    // A22 -= L21 U12 (K = 32): U12 (32 x w2) is staged in shared memory (the caller's buffer
    // past the panel when the panel itself is staged there); each row loads its L21 part and a
    // chunk of its A22 part before storing anything.
    cplx<R>* u12 = sh_u12<R>(sh);
    for (int idx = threadIdx.x; idx < 32 * w2; idx += NT) {
        const int s = idx % 32, q = idx / 32;
        u12[q * 32 + s] = Rt[s + (int64_t)q * ld];
    }
    wsync();
    constexpr int QC = sizeof(R) == 4 ? 16 : 8;  // A22 columns per chunk
    for (int r = w1 + (int)threadIdx.x; r < m; r += NT) {
        cplx<R> lrow[32];
#pragma unroll
        for (int s = 0; s < 32; ++s) lrow[s] = P[r + (int64_t)s * ld];
        for (int q0 = 0; q0 < w2; q0 += QC) {
            cplx<R> x[QC];
#pragma unroll
            for (int j = 0; j < QC; ++j)
                x[j] = (q0 + j < w2) ? Rt[r + (int64_t)(q0 + j) * ld] : czero<R>();
#pragma unroll
            for (int j = 0; j < QC; ++j) {
                if (q0 + j < w2) {
                    const cplx<R>* uq = u12 + (q0 + j) * 32;
#pragma unroll
                    for (int s = 0; s < 32; ++s) cfms(x[j], lrow[s], uq[s]);
                    Rt[r + (int64_t)(q0 + j) * ld] = x[j];
                }
            }
        }
    }
    wsync();
    leaf_factor(Rt + w1, ld, m - w1, w2, sh.piv + w1, col_base + w1, sh);
    if ((int)threadIdx.x < w2) sh.piv[w1 + threadIdx.x] += w1;
    wsync();
    for (int q = threadIdx.x; q < w1; q += NT) {  // right interchanges on the left half
        cplx<R>* cq = P + (int64_t)q * ld;
        for (int c = w1; c < nbk; ++c) {
            const int p = sh.piv[c];
            if (p != c) {
                const cplx<R> t = cq[c];
                cq[c] = cq[p];
                cq[p] = t;
            }
        }
    }
    wsync();
}

// Compose the panel's interchanges (applied in order t = 0..nbk-1) into one permutation of the
// rows they touch.  Entries 0..nbk-1 are the diagonal rows; further entries are pivot rows
// below the panel's diagonal block.  Warp 0 does it; everyone waits.
__device__ void compose_swaps(int nbk, const int* piv, DShared& sh) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        for (int t = lane; t < nbk; t += 32) { sh.rows[t] = t; sh.src[t] = t; }
        __syncwarp();
        int cnt = nbk;
        for (int t = 0; t < nbk; ++t) {
            const int p = piv[t];
            if (p == t) continue;
            int e = -1;
            if (p < nbk) {
                e = p;
            } else {
                for (int base = nbk; base < cnt && e < 0; base += 32) {
                    const int idx = base + lane;
                    const unsigned hit = __ballot_sync(FULL, idx < cnt && sh.rows[idx] == p);
                    if (hit) e = base + __ffs(hit) - 1;
                }
                if (e < 0) {
                    e = cnt;
                    if (lane == 0) { sh.rows[e] = p; sh.src[e] = p; }
                    ++cnt;
                }
            }
            __syncwarp();
            if (lane == 0) {
                const int a = sh.src[t];
                sh.src[t] = sh.src[e];
                sh.src[e] = a;
            }
            __syncwarp();
        }
        if (lane == 0) sh.cnt = cnt;
    }
    wsync();
}

// panel_factor for a panel too tall for shared memory: leaves of lw columns (16, or fewer so that
// m x lw fits), each factored in shared memory; then its interchanges, composed into one permutation, go
// to the panel's other columns, and the columns right of it get their U rows and the rank-lw update.
// The panel's columns cross L2 twice a leaf and column to its right (96 column passes for 64 columns),
// against 1024 when every column of a 32-column leaf updated the others in global memory.
constexpr int kLeafMax = 16;
template <typename R>
__device__ void panel_factor_tall(cplx<R>* P, int64_t ld, int m, int nbk, int lw, int col_base, cplx<R>* sm,
                                  DShared& sh) {
    const int tid = threadIdx.x;
    cplx<R>* u = sh_u12<R>(sh);  // [right column][kLeafMax]
    for (int w0 = 0; w0 < nbk; w0 += lw) {
        const int w = min(lw, nbk - w0), mL = m - w0, nright = nbk - w0 - w, nother = nbk - w;
        cplx<R>* L0 = P + w0 + (int64_t)w0 * ld;
        for (int idx = tid; idx < mL * w; idx += NT) sm[idx] = L0[idx % mL + (int64_t)(idx / mL) * ld];
        wsync();
        leaf_factor(sm, (int64_t)mL, mL, w, sh.piv + w0, col_base + w0, sh);
        compose_swaps(w, sh.piv + w0, sh);
        for (int idx = tid; idx < mL * w; idx += NT) L0[idx % mL + (int64_t)(idx / mL) * ld] = sm[idx];
        const int cnt = sh.cnt;  // at most 2 lw rows are touched
        if (tid < w) sh.piv[w0 + tid] += w0;
        {
            constexpr int MV = 2 * kLeafMax * (NB - kLeafMax) / NT;  // cnt * nother <= 2 lw (NB - lw)
            cplx<R> v[MV];
#pragma unroll
            for (int t = 0; t < MV; ++t) {
                const int idx = tid + NT * t, e = idx % cnt, j = idx / cnt;
                if (j < nother) v[t] = P[(w0 + sh.src[e]) + (int64_t)(j < w0 ? j : j + w) * ld];
            }
            wsync();
#pragma unroll
            for (int t = 0; t < MV; ++t) {
                const int idx = tid + NT * t, e = idx % cnt, j = idx / cnt;
                if (j < nother) P[(w0 + sh.rows[e]) + (int64_t)(j < w0 ? j : j + w) * ld] = v[t];
            }
        }
        wsync();
        if (nright == 0) continue;
        cplx<R>* Rt = P + w0 + (int64_t)(w0 + w) * ld;
        if (tid < nright) {  // U rows: unit lower solve of the leaf's top block
            cplx<R> x[kLeafMax];
#pragma unroll
            for (int r = 0; r < kLeafMax; ++r) x[r] = r < w ? Rt[r + (int64_t)tid * ld] : czero<R>();
#pragma unroll
            for (int r = 1; r < kLeafMax; ++r)
                if (r < w)
#pragma unroll
                    for (int t = 0; t < r; ++t) cfms(x[r], sm[r + t * mL], x[t]);
#pragma unroll
            for (int r = 0; r < kLeafMax; ++r) {
                u[tid * kLeafMax + r] = x[r];
                if (r < w) Rt[r + (int64_t)tid * ld] = x[r];
            }
        }
        wsync();
        constexpr int QC = sizeof(R) == 4 ? 16 : 8;
        for (int r = w + tid; r < mL; r += NT) {
            cplx<R> l[kLeafMax];
#pragma unroll
            for (int t = 0; t < kLeafMax; ++t) l[t] = t < w ? sm[r + t * mL] : czero<R>();
            for (int q0 = 0; q0 < nright; q0 += QC) {
                cplx<R> x[QC];
#pragma unroll
                for (int j = 0; j < QC; ++j)
                    x[j] = (q0 + j < nright) ? Rt[r + (int64_t)(q0 + j) * ld] : czero<R>();
#pragma unroll
                for (int j = 0; j < QC; ++j)
                    if (q0 + j < nright) {
#pragma unroll
                        for (int t = 0; t < kLeafMax; ++t) cfms(x[j], l[t], u[(q0 + j) * kLeafMax + t]);
                        Rt[r + (int64_t)(q0 + j) * ld] = x[j];
                    }
            }
        }
        wsync();
    }
}

// inv(L11) and inv(U11) of the nbk x nbk diagonal block of P; shared layout (r, c) at r * NBP + c:
// sm[0 ..) = inv(L11), then inv(U11), then a copy of the block (its padding column holds 1/U(r,r)).
// Both go to ginv (column-major, leading dimension NB, zero outside nbk x nbk) when `write`.
template <typename R>
__device__ void diag_inverses(const cplx<R>* P, int64_t ld, int nbk, cplx<R>* sm, cplx<R>* ginv, bool write) {
    cplx<R>* iL = sm;
    cplx<R>* iU = sm + NB * NBP;
    cplx<R>* T = sm + 2 * NB * NBP;
    const cplx<R> one = mk<R>(R(1), R(0));
    for (int idx = threadIdx.x; idx < nbk * nbk; idx += NT) {
        const int r = idx % nbk, c = idx / nbk;
        T[r * NBP + c] = P[r + (int64_t)c * ld];
    }
    wsync();
    for (int r = threadIdx.x; r < nbk; r += NT) {
        const cplx<R> d = T[r * NBP + r];
        T[r * NBP + NB] = cis_zero(d) ? czero<R>() : crecip(d);
    }
    wsync();
    const int t = threadIdx.x;
    if (t < nbk) {
        for (int r = 0; r < nbk; ++r) {
            iL[r * NBP + t] = (r == t) ? one : czero<R>();
            iU[r * NBP + t] = czero<R>();
        }
        for (int r = t + 1; r < nbk; ++r) {  // column t of inv(L11): unit lower forward substitution
            cplx<R> a0 = czero<R>(), a1 = czero<R>();
            int s = t;
            for (; s + 1 < r; s += 2) {
                cfms(a0, T[r * NBP + s], iL[s * NBP + t]);
                cfms(a1, T[r * NBP + s + 1], iL[(s + 1) * NBP + t]);
            }
            if (s < r) cfms(a0, T[r * NBP + s], iL[s * NBP + t]);
            iL[r * NBP + t] = a0 + a1;
        }
        iU[t * NBP + t] = T[t * NBP + NB];
        for (int r = t - 1; r >= 0; --r) {  // column t of inv(U11): backward substitution
            cplx<R> a0 = czero<R>(), a1 = czero<R>();
            int s = r + 1;
            for (; s + 1 <= t; s += 2) {
                cfma(a0, T[r * NBP + s], iU[s * NBP + t]);
                cfma(a1, T[r * NBP + s + 1], iU[(s + 1) * NBP + t]);
            }
            if (s <= t) cfma(a0, T[r * NBP + s], iU[s * NBP + t]);
            const cplx<R> acc = a0 + a1;
            iU[r * NBP + t] = mk<R>(-acc.re, -acc.im) * T[r * NBP + NB];
        }
    }
    wsync();
    for (int idx = threadIdx.x; write && idx < NB * NB; idx += NT) {
        const int r = idx % NB, c = idx / NB;
        const bool in = r < nbk && c < nbk;
        ginv[idx] = in ? iL[r * NBP + c] : czero<R>();
        ginv[NB * NB + idx] = in ? iU[r * NBP + c] : czero<R>();
    }
    wsync();
}

// Trailing columns, rows of the panel: apply the composed interchanges and form
// U12 = inv(L11) * (pivot rows), block of TN columns at a time, blocks dealt out over the cluster.
// sm[0..NB*NBP) = inv(L11).
template <typename R>
__device__ void trailing_rows(cplx<R>* A, int64_t lda, int n, int k0, cplx<R>* sm, const DShared& sh,
                              const Cluster& cl) {
    constexpr int TN = DTile<R>::TN;
    const cplx<R>* iL = sm;
    cplx<R>* g = sm + NB * NBP;  // gathered rows, g[col * 2NB + e]
    const int cnt = sh.cnt, extra = cnt - NB;
    for (int c0 = k0 + NB + cl.rank * TN; c0 < n; c0 += cl.size * TN) {
        const int nc = min(TN, n - c0);
        for (int idx = threadIdx.x; idx < cnt * nc; idx += NT) {
            const int e = idx % cnt, col = idx / cnt;
            g[col * 2 * NB + e] = A[(int64_t)(k0 + sh.src[e]) + (int64_t)(c0 + col) * lda];
        }
        wsync();
        for (int idx = threadIdx.x; idx < extra * nc; idx += NT) {
            const int e = NB + idx % extra, col = idx / extra;
            A[(int64_t)(k0 + sh.rows[e]) + (int64_t)(c0 + col) * lda] = g[col * 2 * NB + e];
        }
        {
            // four columns a thread: one entry of inv(L11) and four broadcasts for 16 multiply-adds
            const int t = threadIdx.x % NB, grp = threadIdx.x / NB;
            for (int cb = 4 * grp; cb < nc; cb += 4 * (NT / NB)) {
                const cplx<R>* gc = g + cb * 2 * NB;
                cplx<R> acc[4] = {czero<R>(), czero<R>(), czero<R>(), czero<R>()};
#pragma unroll 4
                for (int s = 0; s <= t; ++s) {
                    const cplx<R> l = iL[t * NBP + s];
#pragma unroll
                    for (int j = 0; j < 4; ++j) cfma(acc[j], l, gc[j * 2 * NB + s]);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (cb + j < nc) A[(int64_t)(k0 + t) + (int64_t)(c0 + cb + j) * lda] = acc[j];
            }
        }
        wsync();
    }
}

// A22 -= L21 * U12 over rows and columns [k0 + NB, n).
template <typename R>
__device__ void trailing_update(cplx<R>* A, int64_t lda, int n, int k0, cplx<R>* sm, const Cluster& cl) {
    using T = DTile<R>;
    constexpr int TM = T::TM, TN = T::TN, MI = T::MI, MJ = T::MJ, TNP = TN + 1;
    cplx<R>* As = sm;                 // [2][NB][TM]
    cplx<R>* Bs = sm + 2 * NB * TM;   // [NB][TNP]
    const int tid = threadIdx.x, ty = tid % 16, tx = tid / 16;
    const int r_begin = k0 + NB;
    const int ntiles = (n - r_begin + TM - 1) / TM;
    const cplx<R>* L21 = A + (int64_t)k0 * lda;  // panel columns
    auto load_a = [&](cplx<R>* buf, int i0) {
        for (int idx = tid; idx < NB * TM; idx += NT) {
            const int r = idx % TM, k = idx / TM;
            const bool ok = i0 + r < n;
            cp_elem(&buf[k * TM + r], ok ? L21 + (i0 + r) + (int64_t)k * lda : A, ok);
        }
    };
    for (int c0 = r_begin + cl.rank * TN; c0 < n; c0 += cl.size * TN) {
        const int ce = min(n, c0 + TN);
        for (int idx = tid; idx < NB * TN; idx += NT) {
            const int k = idx % NB, c = idx / NB;
            const bool ok = c0 + c < ce;
            cp_elem(&Bs[k * TNP + c], ok ? A + (k0 + k) + (int64_t)(c0 + c) * lda : A, ok);
        }
        load_a(As, r_begin);
        cp_commit();
        for (int t = 0; t < ntiles; ++t) {
            const int i0 = r_begin + t * TM;
            if (t + 1 < ntiles) load_a(As + ((t + 1) & 1) * NB * TM, i0 + TM);
            cp_commit();
            cplx<R> acc[MI][MJ];
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < MJ; ++j) {
                    const int r = i0 + ty + 16 * i, c = c0 + tx + 16 * j;
                    acc[i][j] = (r < n && c < ce) ? A[r + (int64_t)c * lda] : czero<R>();
                }
            cp_wait<1>();
            wsync();
            const cplx<R>* Ab = As + (t & 1) * NB * TM;
#pragma unroll 2
            for (int k = 0; k < NB; ++k) {
                cplx<R> a[MI], b[MJ];
#pragma unroll
                for (int i = 0; i < MI; ++i) a[i] = Ab[k * TM + ty + 16 * i];
#pragma unroll
                for (int j = 0; j < MJ; ++j) b[j] = Bs[k * TNP + tx + 16 * j];
#pragma unroll
                for (int i = 0; i < MI; ++i)
#pragma unroll
                    for (int j = 0; j < MJ; ++j) cfms(acc[i][j], a[i], b[j]);
            }
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < MJ; ++j) {
                    const int r = i0 + ty + 16 * i, c = c0 + tx + 16 * j;
                    if (r < n && c < ce) A[r + (int64_t)c * lda] = acc[i][j];
                }
            wsync();
        }
        cp_wait<0>();
        wsync();
    }
}

// ------------------------------------------------------------------------------------------
// Complex64 trailing update on the tensor cores (tcgen05, kind::f16 with BF16 operands).
//
// A22 -= L21 U12 in real arithmetic is four real products (Lr Ur, -Li Ui into the real part;
// Lr Ui, Li Ur into the imaginary part).  Each FP32 operand x is split into three BF16 pieces
// x = h + m + l (h = bf16(x), m = bf16(x - h), l = bf16(x - h - m): 24 significant bits), and a
// product is taken as the six piece products of order >= 2^-16 (hh, hm, mh, hl, mm, lh) with
// FP32 accumulation in tensor memory: FP32-level accuracy (what is dropped is ~2^-24 relative).
// The FP64 refinement of the sample solves sits on top as for the CUDA-core path.  Against a
// two-piece TF32 split (three products) this is the same tensor time, but the operands take
// 12 instead of 16 bytes per complex value, which lets a 128 x 128 step fit in shared memory:
// N = 128 per MMA keeps the operand reads per MMA within the shared-memory bandwidth.
//
// Per panel the operands are split once into "images" in global memory whose bytes are exactly
// the shared-memory layout the MMA reads (K-major, 128-byte swizzle, K = 64 = one 128-byte row):
// one 96 KB image per 128-row tile of L21 and one per 128-column block of U12.  For each L21
// tile the MMA issuer (thread 0) bulk-copies the tile, then walks the U12 blocks through one smem
// buffer and two TMEM accumulator pairs: while all 8 warps run the epilogue of block t (C
// prefetched from global memory, TMEM -> registers, C -= D), thread 0 refills the buffer with
// block t+1 and issues its MMAs.  Every wait is bounded; a timeout marks the job failed.
// ------------------------------------------------------------------------------------------
struct TcShared {
    // 0: L21 tile; 1: U12 buffer; 2: command to the producer warp; 3 + b: epilogue of accumulator
    // pair b done (one arrival per worker warp); 5 + b: MMAs into accumulator pair b done
    uint64_t bar[7];
    uint32_t tmem;       // tensor-memory base address
    int fail;            // set by any thread whose bounded wait ran out
    int stop;            // the workers' common view of `fail`, written by worker thread 0 between barriers
    int cmd;             // 1: run a trailing update with the parameters below, 2: exit
    int n, k0;
    int64_t lda;
    const float* imgA;
    const float* imgB;
    int rank, size;      // of the cluster: step g of an update is CTA g % size's
};
struct TcPhase {
    uint32_t a = 0, b = 0, go = 0, e[2] = {0, 0}, d[2] = {0, 0};
};

__device__ __forceinline__ bool failed(const TcShared& ts) { return *(const volatile int*)&ts.fail != 0; }

// Write the six BF16 pieces of v[0..8) at (row r, k..k+7) of an operand image with `rows` rows: array q
// (0..2 re hi/mid/lo, 3..5 im hi/mid/lo) occupies rows * 64 elements.  Eight consecutive k are one
// 16-byte unit of the swizzled layout.
__device__ __forceinline__ void put_split8(float* img, int r, int k, int rows, const c64* v) {
    unsigned char* t = reinterpret_cast<unsigned char*>(img) + sw128_index16(r, k) * 2;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        __align__(16) __nv_bfloat16 h[8], m[8], l[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float x = c ? v[e].im : v[e].re;
            h[e] = __float2bfloat16_rn(x);
            const float r1 = x - __bfloat162float(h[e]);
            m[e] = __float2bfloat16_rn(r1);
            l[e] = __float2bfloat16_rn(r1 - __bfloat162float(m[e]));
        }
        const size_t stride = (size_t)rows * NB * 2;
        *reinterpret_cast<uint4*>(t + (3 * c + 0) * stride) = *reinterpret_cast<const uint4*>(h);
        *reinterpret_cast<uint4*>(t + (3 * c + 1) * stride) = *reinterpret_cast<const uint4*>(m);
        *reinterpret_cast<uint4*>(t + (3 * c + 2) * stride) = *reinterpret_cast<const uint4*>(l);
    }
}

// L21 (rows k0+NB.., panel columns) -> one image per 128-row tile; rows past n are zero.
__device__ void emit_a_image(const c64* A, int64_t lda, int n, int k0, float* img, const Cluster& cl) {
    const int r_begin = k0 + NB, m = n - r_begin;
    const int rows_pad = (m + TC_ROWS - 1) / TC_ROWS * TC_ROWS;
    for (int idx = cl.rank * NT + threadIdx.x; idx < rows_pad * (NB / 8); idx += cl.size * NT) {
        const int rr = idx % rows_pad, k = idx / rows_pad * 8;
        c64 v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            v[e] = rr < m ? A[(int64_t)(r_begin + rr) + (int64_t)(k0 + k + e) * lda] : czero<float>();
        put_split8(img + (size_t)(rr / TC_ROWS) * TC_A_FLOATS, rr % TC_ROWS, k, TC_ROWS, v);
    }
}
// U12 (panel rows, columns k0+NB..) -> one image per 128-column block (the CTA's own blocks, whose
// U12 it has just formed); columns past n are zero.
__device__ void emit_b_image(const c64* A, int64_t lda, int n, int k0, float* img, const Cluster& cl) {
    static_assert(TC_COLS == (uint32_t)DTile<float>::TN, "a CTA's U12 blocks are its image blocks");
    const int c_begin = k0 + NB, m = n - c_begin;
    const int nblk = (m + TC_COLS - 1) / TC_COLS, own = (nblk - cl.rank + cl.size - 1) / cl.size;
    for (int idx = threadIdx.x; idx < own * (int)TC_COLS * (NB / 8); idx += NT) {
        const int k = idx % (NB / 8) * 8, q = idx / (NB / 8);
        const int cc = (cl.rank + q / TC_COLS * cl.size) * TC_COLS + q % TC_COLS;
        c64 v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            v[e] = cc < m ? A[(int64_t)(k0 + k + e) + (int64_t)(c_begin + cc) * lda] : czero<float>();
        put_split8(img + (size_t)(cc / TC_COLS) * TC_B_FLOATS, cc % TC_COLS, k, TC_COLS, v);
    }
}

// All MMAs of one (L21 tile, U12 block) step into the accumulator pair at TMEM column dt:
// re part at dt, im part at dt + 128.  Descriptors are built once; an offset of o bytes inside
// an operand buffer is + (o >> 4) on the descriptor (no carry: the buffers lie below 256 KB).
__device__ __forceinline__ void tc_issue(uint64_t adesc, uint64_t bdesc, uint32_t dt) {
    // kind::f16: F32 accumulate, BF16 A and B, K-major both, N = 128, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((TC_COLS >> 3) << 17) | ((TC_ROWS >> 4) << 24);
    const int pa[4] = {0, 1, 0, 1}, pb[4] = {0, 1, 1, 0}, pd[4] = {0, 0, 128, 128}, ng[4] = {0, 1, 0, 0};
    const int sa[6] = {0, 0, 1, 0, 1, 2}, sb[6] = {0, 1, 0, 2, 1, 0};  // hh hm mh hl mm lh
    uint32_t acc_r = 0, acc_i = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t id = idesc | (ng[p] ? (1u << 13) : 0u);  // negate A for -Li Ui
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            const uint32_t qa = pa[p] * TC_SPLIT + sa[s], qb = pb[p] * TC_SPLIT + sb[s];
#pragma unroll
            for (int ks = 0; ks < NB / 16; ++ks) {
                const uint32_t ao = qa * TC_ROWS * NB * 2 + ks * 32;
                const uint32_t bo = qb * TC_COLS * NB * 2 + ks * 32;
                uint32_t& acc = pd[p] ? acc_i : acc_r;
                tc_mma(dt + pd[p], adesc + (ao >> 4), bdesc + (bo >> 4), id, acc);
                acc = 1;
            }
        }
    }
}

// C -= D for one 128 x 128 step: warp w reads TMEM lanes 32 (w % 4).., complex columns 64 (w / 4)..
// in two chunks of 32.  `v` holds a chunk of C values, loaded before the TMEM data is waited for.
__device__ __forceinline__ void tc_load_c(const c64* A, int64_t lda, int n, int i0, int c0, int chunk, c64* v) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, half = warp >> 2;
    const int row = i0 + 32 * q + lane, cb = c0 + half * 64 + chunk * 32;
#pragma unroll
    for (int c = 0; c < 32; ++c)
        v[c] = (row < n && cb + c < n) ? A[row + (int64_t)(cb + c) * lda] : czero<float>();
}
__device__ __forceinline__ void tc_store_c(c64* A, int64_t lda, int n, int i0, int c0, int chunk, uint32_t tbuf,
                                           const c64* v) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, half = warp >> 2;
    const uint32_t ta = tbuf + ((uint32_t)(32 * q) << 16) + (uint32_t)(half * 64 + chunk * 32);
    const int row = i0 + 32 * q + lane, cb = c0 + half * 64 + chunk * 32;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float dr[16], di[16];
        tc_ld16(ta + h * 16, dr);
        tc_ld16(ta + 128 + h * 16, di);
        tc_wait_ld();
        if (row < n) {
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const int col = cb + h * 16 + c;
                if (col < n) A[row + (int64_t)col * lda] = mk<float>(v[h * 16 + c].re - dr[c], v[h * 16 + c].im - di[c]);
            }
        }
    }
}

// Worker side (warps 0..7) of one panel's trailing update: hand the parameters to the producer
// warp, then for every (L21 tile, U12 block) step in order: prefetch C, wait for the step's
// MMAs, read the accumulators, release them to the producer, write C back.
__device__ void trailing_update_tc(c64* A, int64_t lda, int n, int k0, const float* imgA, const float* imgB,
                                   TcShared& ts, TcPhase& ph) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int r_begin = k0 + NB, m = n - r_begin;
    const int ncb = (m + TC_COLS - 1) / TC_COLS, steps = (m + TC_ROWS - 1) / TC_ROWS * ncb;
    if (tid == 0) {
        ts.n = n;
        ts.k0 = k0;
        ts.lda = lda;
        ts.imgA = imgA;
        ts.imgB = imgB;
        ts.cmd = 1;
        mbar_arrive(&ts.bar[2]);  // release: the producer reads the parameters after its wait
    }
    c64 v[32];
    for (int g = ts.rank, i = 0; g < steps && !failed(ts); g += ts.size, ++i) {
        const int b = i & 1;
        const int i0 = r_begin + (g / ncb) * TC_ROWS, c0 = r_begin + (g % ncb) * TC_COLS;
        const uint32_t tb = ts.tmem + b * 256;
        tc_load_c(A, lda, n, i0, c0, 0, v);
        if (!mbar_wait(&ts.bar[5 + b], ph.d[b])) ts.fail = 1;
        ph.d[b] ^= 1;
        tc_fence_after();
        tc_store_c(A, lda, n, i0, c0, 0, tb, v);
        tc_load_c(A, lda, n, i0, c0, 1, v);
        tc_store_c(A, lda, n, i0, c0, 1, tb, v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ts.bar[3 + b]);
    }
    wsync();  // warps may leave the loop at different steps after a timeout; all meet here
    if (tid == 0) ts.stop = failed(ts) ? 1 : 0;
    wsync();
}

// Producer warp (warp 8; lane 0 issues): per trailing update, bulk-copy each L21 tile and U12
// block into shared memory and issue the step's MMAs into accumulator pair g % 2 once the
// workers have released it.  Runs until the exit command.
__device__ void tc_producer(unsigned char* smem_raw, TcShared& ts) {
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sB = base + TC_A_BYTES;
    const uint64_t adesc = sw128_desc(smem_u32(base)), bdesc = sw128_desc(smem_u32(sB));
    const bool leader = (threadIdx.x & 31) == 0;
    uint32_t pa = 0, pb = 0, pgo = 0, pm[2] = {0, 0}, pe[2] = {0, 0};
    auto wait = [&](uint64_t* bar, uint32_t& par) {
        if (!failed(ts) && !mbar_wait(bar, par)) ts.fail = 1;
        par ^= 1;
    };
    for (;;) {
        // the command barrier completes once per command; the workers factor a panel in between,
        // so one bounded wait may run out: retry a bounded number of times, then give up
        int got = 0;
        if (leader)
            for (int tries = 0; tries < 64 && !got; ++tries) got = mbar_wait(&ts.bar[2], pgo) ? 1 : 0;
        got = __shfl_sync(FULL, got, 0);  // one decision for the whole warp
        if (!got) {
            ts.fail = 1;
            return;
        }
        pgo ^= 1;
        if (*(volatile int*)&ts.cmd != 1) break;
        const int n = *(volatile int*)&ts.n, k0 = *(volatile int*)&ts.k0;
        const float* imgA = *(const float* volatile*)&ts.imgA;
        const float* imgB = *(const float* volatile*)&ts.imgB;
        const int r_begin = k0 + NB, m = n - r_begin;
        const int ncb = (m + TC_COLS - 1) / TC_COLS, steps = (m + TC_ROWS - 1) / TC_ROWS * ncb;
        const int mine = steps > ts.rank ? (steps - ts.rank + ts.size - 1) / ts.size : 0;
        for (int i = 0, prev_rt = -1; i < mine; ++i) {
            const int g = ts.rank + i * ts.size, rt = g / ncb, t = g % ncb, b = i & 1;
            const bool new_a = rt != prev_rt;  // L21 tile to load
            prev_rt = rt;
            if (i > 0) wait(&ts.bar[5 + ((i - 1) & 1)], pm[(i - 1) & 1]);  // the operand buffers are free
            if (leader && !failed(ts)) {
                if (new_a) {
                    mbar_expect_tx(&ts.bar[0], TC_A_BYTES);
                    for (int c = 0; c < 6; ++c)
                        bulk_g2s(base + c * (TC_A_BYTES / 6), imgA + (size_t)rt * TC_A_FLOATS + c * (TC_A_FLOATS / 6),
                                 TC_A_BYTES / 6, &ts.bar[0]);
                }
                mbar_expect_tx(&ts.bar[1], TC_B_BYTES);
                const float* src = imgB + (size_t)t * TC_B_FLOATS;
                for (int c = 0; c < 6; ++c)
                    bulk_g2s(sB + c * (TC_B_BYTES / 6), src + c * (TC_B_FLOATS / 6), TC_B_BYTES / 6, &ts.bar[1]);
                if (i + 1 < mine) {
                    const int gn = g + ts.size;
                    prefetch_l2(imgB + (size_t)(gn % ncb) * TC_B_FLOATS, TC_B_BYTES);
                    if (gn / ncb != rt) prefetch_l2(imgA + (size_t)(gn / ncb) * TC_A_FLOATS, TC_A_BYTES);
                }
            }
            __syncwarp();
            if (new_a) wait(&ts.bar[0], pa);
            wait(&ts.bar[1], pb);
            if (i >= 2) wait(&ts.bar[3 + b], pe[b]);  // the workers have read accumulator pair b
            tc_fence_after();
            if (leader) {
                if (!failed(ts)) tc_issue(adesc, bdesc, ts.tmem + b * 256);
                tc_commit(&ts.bar[5 + b]);
            }
            __syncwarp();
        }
        // consume the completions not waited for above, so every barrier's phase stays in step
        if (mine > 0) wait(&ts.bar[5 + ((mine - 1) & 1)], pm[(mine - 1) & 1]);
        if (mine > 1) wait(&ts.bar[3 + ((mine - 2) & 1)], pe[(mine - 2) & 1]);
        if (mine > 0) wait(&ts.bar[3 + ((mine - 1) & 1)], pe[(mine - 1) & 1]);
    }
}

// The panel is CTA 0's; U12's column blocks, the images and the update's steps are dealt out over the
// cluster.  sh.info is the same in every CTA after the barrier that follows a panel.
template <typename R>
__device__ void factor_one(const DenseJob<R>& J, cplx<R>* sm, DShared& sh, float* img, size_t img_b, TcShared* ts,
                           TcPhase* ph, Cluster& cl) {
    const int n = J.n;
    const int64_t lda = J.lda;
    cplx<R>* A = J.a;
    const int cap_rows = (int)(factor_smem<R>() / (NB * sizeof(cplx<R>)));
    for (int p = 0, k0 = 0; k0 < n; ++p, k0 += NB) {
        const int nbk = min(NB, n - k0), m = n - k0;
        cplx<R>* Pg = A + k0 + (int64_t)k0 * lda;
        int32_t* sw = J.swaps + (int64_t)p * kDenseSwapInts;
        if (cl.rank == 0) {
            if (m <= cap_rows) {
                for (int idx = threadIdx.x; idx < m * nbk; idx += NT) {
                    const int r = idx % m, c = idx / m;
                    sm[r + c * m] = Pg[r + (int64_t)c * lda];
                }
                wsync();
                panel_factor(sm, (int64_t)m, m, nbk, k0, sh);
                for (int idx = threadIdx.x; idx < m * nbk; idx += NT) {
                    const int r = idx % m, c = idx / m;
                    Pg[r + (int64_t)c * lda] = sm[r + c * m];
                }
                wsync();
            } else {
                int lw = kLeafMax;
                while (lw > 2 && (size_t)m * lw * sizeof(cplx<R>) > factor_smem<R>()) lw /= 2;
                // leaves of fewer than 4 columns would cross L2 as often as the columns themselves
                if (lw >= 4) panel_factor_tall(Pg, lda, m, nbk, lw, k0, sm, sh);
                else panel_factor(Pg, lda, m, nbk, k0, sh);
            }
            if ((int)threadIdx.x < nbk) J.ipiv[k0 + threadIdx.x] = k0 + sh.piv[threadIdx.x];
            compose_swaps(nbk, sh.piv, sh);
            if (threadIdx.x == 0) sw[0] = sh.cnt;
            for (int i = threadIdx.x; i < 2 * NB; i += NT) {
                sw[1 + i] = i < sh.cnt ? sh.rows[i] : 0;
                sw[1 + 2 * NB + i] = i < sh.cnt ? sh.src[i] : 0;
            }
            if ((int)threadIdx.x < cl.size && threadIdx.x > 0)
                *cg::this_cluster().map_shared_rank(&sh.info, threadIdx.x) = sh.info;
        }
        if (!csync(cl, sh)) { sh.info = -1; break; }
        if (cl.rank != 0) {
            if (threadIdx.x == 0) sh.cnt = __ldcg(sw);
            for (int i = threadIdx.x; i < 2 * NB; i += NT) {
                sh.rows[i] = __ldcg(sw + 1 + i);
                sh.src[i] = __ldcg(sw + 1 + 2 * NB + i);
            }
            wsync();
        }
        diag_inverses(Pg, lda, nbk, sm, J.inv + (int64_t)p * 2 * NB * NB, cl.rank == 0);
        if (k0 + nbk < n) {
            trailing_rows(A, lda, n, k0, sm, sh, cl);
            if constexpr (sizeof(R) == 4) {
                emit_a_image(A, lda, n, k0, img, cl);
                emit_b_image(A, lda, n, k0, img + img_b, cl);
                // the images (global) and the shared buffers were last touched through the generic
                // proxy; the bulk copies and MMAs that follow go through the async proxy
                asm volatile("fence.proxy.async.global;" ::: "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (!csync(cl, sh)) { sh.info = -1; break; }
                asm volatile("fence.proxy.async.global;" ::: "memory");
                trailing_update_tc(A, lda, n, k0, img, img + img_b, *ts, *ph);
                if (ts->stop) {  // uniform: written by thread 0 between two worker barriers
                    sh.info = -1;
                    cluster_fail(cl, sh);
                    break;
                }
            } else {
                if (!csync(cl, sh)) { sh.info = -1; break; }
                trailing_update(A, lda, n, k0, sm, cl);
            }
        }
        if (!csync(cl, sh)) { sh.info = -1; break; }
    }
}

// ------------------------------------------------------------------------------------------
// Solves.  x (n x L, leading dimension n) <- A^{-1} x.  Forward: per panel, the composed
// interchanges, y = inv(L11) x_top, x_below -= L21 y.  Backward: per panel from the last,
// y = inv(U11) x_top, x_above -= U01 y.  Right-hand sides in groups of LG columns.
// ------------------------------------------------------------------------------------------
constexpr int LG = 32;  // right-hand-side columns per pass over the factor
template <typename R> struct SolveChunk;
template <> struct SolveChunk<float> { static constexpr int LC = 8; };
template <> struct SolveChunk<double> { static constexpr int LC = 4; };

template <typename R>
constexpr size_t solve_smem() {
    return ((size_t)NB * NBP + (size_t)2 * NB * LG + (size_t)NB * LG) * sizeof(cplx<R>);
}

// x[r, l] -= sum_k Ablk[r + k lda] y[k * LP + l]  for r in [r0, r1), l < lg
template <typename R, int LC>
__device__ void solve_update(const cplx<R>* Ablk, int64_t lda, int r0, int r1, int nbk,
                             const cplx<R>* y, int LP, int lg, cplx<R>* x, int64_t ldx) {
    for (int l0 = 0; l0 < lg; l0 += LC) {
        for (int r = r0 + (int)threadIdx.x; r < r1; r += NT) {
            cplx<R> acc[LC];
#pragma unroll
            for (int l = 0; l < LC; ++l) acc[l] = (l0 + l < lg) ? x[r + (int64_t)(l0 + l) * ldx] : czero<R>();
            // the factor's entries of 32 columns in flight: the pass is bound by the latency of L2
#pragma unroll 32
            for (int k = 0; k < nbk; ++k) {
                const cplx<R> a = Ablk[r + (int64_t)k * lda];
#pragma unroll
                for (int l = 0; l < LC; ++l) cfms(acc[l], a, y[k * LP + l0 + l]);
            }
#pragma unroll
            for (int l = 0; l < LC; ++l)
                if (l0 + l < lg) x[r + (int64_t)(l0 + l) * ldx] = acc[l];
        }
    }
}

// x <- A^{-1} x for one factored point (columns l_lo .. l_hi - 1), by the NT worker threads.
// smem: solve_smem<R>() bytes; rows/src/cnt: 2 NB + 2 NB + 1 ints of shared scratch.
template <typename R>
__device__ void solve_one(const DenseJob<R>& J, int l_lo, int l_hi, unsigned char* smem, int* s_rows, int* s_src,
                          int* s_cnt) {
    constexpr int LC = SolveChunk<R>::LC;
    cplx<R>* sinv = reinterpret_cast<cplx<R>*>(smem);  // (r, c) at r * NBP + c
    cplx<R>* g = sinv + NB * NBP;                      // [2 NB][LG]
    cplx<R>* y = g + 2 * NB * LG;                      // [NB][LP]
    const int n = J.n;
    const int np = (int)dense_panels(n);
    const int64_t lda = J.lda;
    auto update = [&](const cplx<R>* Ablk, int r0, int r1, int nbk, const cplx<R>* y, int LP, int lg, cplx<R>* x) {
        if (lg <= 2) solve_update<R, 2>(Ablk, lda, r0, r1, nbk, y, LP, lg, x, n);
        else solve_update<R, LC>(Ablk, lda, r0, r1, nbk, y, LP, lg, x, n);
    };
    for (int l_begin = l_lo; l_begin < l_hi; l_begin += LG) {
        const int lg = min(LG, l_hi - l_begin);
        const int LP = (lg + LC - 1) / LC * LC;
        cplx<R>* x = J.x + (int64_t)l_begin * n;
        for (int idx = threadIdx.x; idx < NB * LP; idx += NT) y[idx] = czero<R>();
        wsync();
        for (int p = 0; p < np; ++p) {  // forward
            const int k0 = p * NB, nbk = min(NB, n - k0);
            const int32_t* sw = J.swaps + (int64_t)p * kDenseSwapInts;
            const cplx<R>* gi = J.inv + (int64_t)p * 2 * NB * NB;
            if (threadIdx.x == 0) *s_cnt = sw[0];
            for (int i = threadIdx.x; i < 2 * NB; i += NT) {
                s_rows[i] = sw[1 + i];
                s_src[i] = sw[1 + 2 * NB + i];
            }
            for (int idx = threadIdx.x; idx < nbk * nbk; idx += NT) {
                const int r = idx % nbk, c = idx / nbk;
                sinv[r * NBP + c] = gi[r + c * NB];
            }
            wsync();
            const int cnt = *s_cnt;
            for (int idx = threadIdx.x; idx < cnt * lg; idx += NT) {
                const int e = idx % cnt, l = idx / cnt;
                g[e * LG + l] = x[k0 + s_src[e] + (int64_t)l * n];
            }
            wsync();
            const int extra = cnt - nbk;
            for (int idx = threadIdx.x; idx < extra * lg; idx += NT) {
                const int e = nbk + idx % extra, l = idx / extra;
                x[k0 + s_rows[e] + (int64_t)l * n] = g[e * LG + l];
            }
            for (int idx = threadIdx.x; idx < nbk * lg; idx += NT) {
                const int t = idx % nbk, l = idx / nbk;
                cplx<R> acc = czero<R>();
                for (int s = 0; s <= t; ++s) cfma(acc, sinv[t * NBP + s], g[s * LG + l]);
                y[t * LP + l] = acc;
                x[k0 + t + (int64_t)l * n] = acc;
            }
            wsync();
            if (k0 + nbk < n) update(J.a + (int64_t)k0 * lda, k0 + nbk, n, nbk, y, LP, lg, x);
            wsync();
        }
        for (int p = np - 1; p >= 0; --p) {  // backward
            const int k0 = p * NB, nbk = min(NB, n - k0);
            const cplx<R>* gi = J.inv + (int64_t)p * 2 * NB * NB + NB * NB;
            for (int idx = threadIdx.x; idx < nbk * nbk; idx += NT) {
                const int r = idx % nbk, c = idx / nbk;
                sinv[r * NBP + c] = gi[r + c * NB];
            }
            for (int idx = threadIdx.x; idx < nbk * lg; idx += NT) {
                const int t = idx % nbk, l = idx / nbk;
                g[t * LG + l] = x[k0 + t + (int64_t)l * n];
            }
            wsync();
            for (int idx = threadIdx.x; idx < nbk * lg; idx += NT) {
                const int t = idx % nbk, l = idx / nbk;
                cplx<R> acc = czero<R>();
                for (int s = t; s < nbk; ++s) cfma(acc, sinv[t * NBP + s], g[s * LG + l]);
                y[t * LP + l] = acc;
                x[k0 + t + (int64_t)l * n] = acc;
            }
            wsync();
            if (k0 > 0) update(J.a + (int64_t)k0 * lda, 0, k0, nbk, y, LP, lg, x);
            wsync();
        }
    }
}

// ------------------------------------------------------------------------------------------
// Fused dense sampling.  Per job (point j of NEP E), in the cluster's slot:
//   zero the matrix, scatter T(z_j) = sum_i f_i(z_j) A_i (precision R) and the FP64 column
//   sums |T| (for ||T||_1); factor; x = U; solve; X = x in S_hat (FP64); then
//   r = U - T X in FP64 from T's CSR values (kept from the assembly, or recomputed), eta per column,
//   and refinement X += (LU)^{-1} r while the stopping rule of the band path asks for it.
// ------------------------------------------------------------------------------------------
constexpr int kMaxL = 256;

constexpr int kMaxCluster = 8;

struct SampleShared {
    double rn2[kMaxL], xn2[kMaxL];
    double red[NW];
    double normT, mx;
    int action;
};

template <typename R>
struct Slot {
    cplx<R>* a;
    cplx<R>* x;
    int32_t* ipiv;
    cplx<R>* inv;
    int32_t* swaps;
    double* colsum;
    c128* tv;      // T(z_j) on the CSR pattern, or null
    double* part;  // [kMaxCluster][2][L] the CTAs' shares of the residual's sums
};

__host__ __device__ inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

template <typename R>
__host__ __device__ inline size_t slot_bytes(int n_max, int L_max, int64_t nnz_max) {
    const size_t np = (size_t)dense_panels(n_max);
    return align256((size_t)n_max * n_max * sizeof(cplx<R>)) + align256((size_t)n_max * L_max * sizeof(cplx<R>)) +
           align256((size_t)n_max * 4) + align256(np * 2 * NB * NB * sizeof(cplx<R>)) +
           align256(np * kDenseSwapInts * 4) + align256((size_t)n_max * 8) + align256((size_t)nnz_max * sizeof(c128)) +
           align256((size_t)kMaxCluster * 2 * L_max * sizeof(double));
}

template <typename R>
__device__ Slot<R> slot_at(unsigned char* base, int n_max, int L_max, int64_t nnz_max) {
    const size_t np = (size_t)dense_panels(n_max);
    Slot<R> t;
    unsigned char* p = base;
    t.a = reinterpret_cast<cplx<R>*>(p);
    p += align256((size_t)n_max * n_max * sizeof(cplx<R>));
    t.x = reinterpret_cast<cplx<R>*>(p);
    p += align256((size_t)n_max * L_max * sizeof(cplx<R>));
    t.ipiv = reinterpret_cast<int32_t*>(p);
    p += align256((size_t)n_max * 4);
    t.inv = reinterpret_cast<cplx<R>*>(p);
    p += align256(np * 2 * NB * NB * sizeof(cplx<R>));
    t.swaps = reinterpret_cast<int32_t*>(p);
    p += align256(np * kDenseSwapInts * 4);
    t.colsum = reinterpret_cast<double*>(p);
    p += align256((size_t)n_max * 8);
    t.tv = nnz_max > 0 ? reinterpret_cast<c128*>(p) : nullptr;
    p += align256((size_t)nnz_max * sizeof(c128));
    t.part = reinterpret_cast<double*>(p);
    return t;
}

// Block-wide max of one double per thread (workers only); every worker gets the result.
__device__ double worker_max(double v, SampleShared& ss) {
    for (int off = 16; off; off >>= 1) v = fmax(v, __shfl_down_sync(FULL, v, off));
    if ((threadIdx.x & 31) == 0) ss.red[threadIdx.x >> 5] = v;
    wsync();
    double m = ss.red[0];
    for (int w = 1; w < NW; ++w) m = fmax(m, ss.red[w]);
    wsync();
    return m;
}

// r = U - T X (FP64, T's CSR values tv if KEPT, else formed from the terms); x = r in precision R; per-column ||r||^2 and ||X||^2 into
// ss.rn2 / ss.xn2 (this CTA's rows only).  A warp takes a row: lane = (column of a group of 8, one of 4 entries), so that no
// lane idles; the FP64 rate bounds it (two multiply-adds a clock: 1 ms for 132000 entries and 8
// columns, where a thread a row and T formed anew from its terms took 2.7 ms).
template <typename R, bool KEPT>
__device__ void residual_one(const DenseNep& E, int j, const c128* X, const c128* tv, cplx<R>* x, SampleShared& ss,
                             const Cluster& cl) {
    const int n = E.n, L = E.L, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 3;
    for (int l = threadIdx.x; l < L; l += NT) ss.rn2[l] = ss.xn2[l] = 0.0;
    wsync();
    for (int l0 = 0; l0 < L; l0 += 8) {
        const int l = l0 + (lane & 7);
        const bool on = l < L;
        const c128* Xl = X + (int64_t)(on ? l : l0) * n;
        double pr = 0.0, px = 0.0;
        for (int r = cl.rank * NW + warp; r < n; r += cl.size * NW) {
            const int64_t end = E.rowptr[r + 1];
            c128 acc = czero<double>();
            if constexpr (KEPT) {
#pragma unroll 4
                for (int64_t k = E.rowptr[r] + sub; k < end; k += 4) cfma(acc, tv[k], Xl[E.colind[k]]);
            } else {
                const c128* f = E.F + (int64_t)j * E.J;
                for (int64_t k = E.rowptr[r] + sub; k < end; k += 4) {
                    c128 t = czero<double>();
                    for (int i = 0; i < E.J; ++i) cfma(t, f[i], E.vals[(int64_t)i * E.nnz + k]);
                    cfma(acc, t, Xl[E.colind[k]]);
                }
            }
#pragma unroll
            for (int off = 8; off <= 16; off <<= 1) {
                acc.re += __shfl_xor_sync(FULL, acc.re, off);
                acc.im += __shfl_xor_sync(FULL, acc.im, off);
            }
            if (sub == 0 && on) {
                const c128 res = E.U[r + (int64_t)l * n] - acc;
                x[r + (int64_t)l * n] = ccast<R>(res);
                pr += cnorm2(res);
                px += cnorm2(Xl[r]);
            }
        }
        if (sub == 0 && on) {
            atomicAdd(&ss.rn2[l], pr);
            atomicAdd(&ss.xn2[l], px);
        }
    }
    wsync();
}

template <typename R, bool KEPT>
__device__ void sample_one(const DenseNep& E, int j, const Slot<R>& sl, cplx<R>* sm, DShared& sh, SampleShared& ss,
                           float* img, size_t img_b, TcShared* ts, TcPhase* ph, const DenseSampleCfg& cfg, Cluster& cl) {
    const int n = E.n, L = E.L, J = E.J;
    const int64_t nnz = E.nnz, nl = (int64_t)n * L;
    const int gtid = cl.rank * NT + threadIdx.x, gstep = cl.size * NT;
    const int l_lo = L * cl.rank / cl.size, l_hi = L * (cl.rank + 1) / cl.size;  // this CTA's columns
    const int64_t x_lo = (int64_t)n * l_lo, x_hi = (int64_t)n * l_hi;
    cplx<R>* A = sl.a;
    auto failed_wait = [&]() {  // a wait in the cluster gave up: every CTA that notices reports the point
        if (threadIdx.x == 0) {
            E.status[j] = -1;
            E.sweeps[j] = 0;
        }
        wsync();
    };
    // assemble T(z_j) (precision R) and its FP64 column sums
    {
        const int64_t nn = (int64_t)n * n;
        for (int64_t idx = gtid; idx < nn; idx += gstep) A[idx] = czero<R>();
        for (int c = gtid; c < n; c += gstep) sl.colsum[c] = 0.0;
        if (!csync(cl, sh)) return failed_wait();
        const c128* f = E.F + (int64_t)j * J;
        for (int64_t k = gtid; k < nnz; k += gstep) {
            c128 t = czero<double>();
            for (int i = 0; i < J; ++i) cfma(t, f[i], E.vals[(int64_t)i * nnz + k]);
            if constexpr (KEPT) sl.tv[k] = t;
            const int c = E.colind[k];
            A[E.rowidx[k] + (int64_t)c * n] = ccast<R>(t);
            atomicAdd(&sl.colsum[c], sqrt(cnorm2(t)));
        }
        if (threadIdx.x == 0) sh.info = 0;
        if (!csync(cl, sh)) return failed_wait();
        double m = 0.0;
        for (int c = threadIdx.x; c < n; c += NT) m = fmax(m, __ldcg(sl.colsum + c));
        m = worker_max(m, ss);
        if (threadIdx.x == 0) ss.normT = m;
    }
    DenseJob<R> Jb;
    Jb.a = A;
    Jb.lda = n;
    Jb.n = n;
    Jb.L = L;
    Jb.ipiv = sl.ipiv;
    Jb.inv = sl.inv;
    Jb.swaps = sl.swaps;
    Jb.x = sl.x;
    factor_one(Jb, sm, sh, img, img_b, ts, ph, cl);
    wsync();
    const int info = sh.info;
    if (info < 0) return failed_wait();
    if (info != 0) {
        if (threadIdx.x == 0 && cl.rank == 0) {
            E.status[j] = info;
            E.sweeps[j] = 0;
        }
        wsync();
        return;
    }
    c128* X = E.S + (int64_t)j * nl;
    for (int64_t idx = x_lo + threadIdx.x; idx < x_hi; idx += NT) sl.x[idx] = ccast<R>(E.U[idx]);
    wsync();
    unsigned char* smb = reinterpret_cast<unsigned char*>(sm);
    solve_one(Jb, l_lo, l_hi, smb, sh.rows, sh.src, &sh.cnt);
    for (int64_t idx = x_lo + threadIdx.x; idx < x_hi; idx += NT) X[idx] = ccast<double>(sl.x[idx]);
    double prev = 0.0;
    int sweeps = 0;
    for (;;) {
        if (!csync(cl, sh)) return failed_wait();  // every column of X is there
        residual_one<R, KEPT>(E, j, X, sl.tv, sl.x, ss, cl);
        for (int l = threadIdx.x; l < L; l += NT) {
            sl.part[(2 * cl.rank) * L + l] = ss.rn2[l];
            sl.part[(2 * cl.rank + 1) * L + l] = ss.xn2[l];
        }
        if (!csync(cl, sh)) return failed_wait();
        // backward error per column and the decision (the same in every CTA: the same sums)
        double mx = 0.0;
        int nonfinite = 0;
        for (int l = threadIdx.x; l < L; l += NT) {
            double rn2 = 0.0, xn2 = 0.0;
            for (int q = 0; q < cl.size; ++q) {
                rn2 += __ldcg(sl.part + (2 * q) * L + l);
                xn2 += __ldcg(sl.part + (2 * q + 1) * L + l);
            }
            const double e = sqrt(rn2) / (ss.normT * sqrt(xn2) + sqrt(E.un2[l]));
            if (cl.rank == 0) E.eta[(int64_t)j * L + l] = e;
            if (!isfinite(e)) nonfinite = 1;
            mx = fmax(mx, e);
        }
        mx = worker_max(nonfinite ? INFINITY : mx, ss);
        if (threadIdx.x == 0) {
            int action;                                          // 0 done, 1 refine, < 0 failed
            const bool improving = sweeps == 0 || mx < 0.5 * prev;
            if (!isfinite(mx)) action = -2;
            else if (!(mx <= cfg.target) && improving) action = sweeps >= cfg.max_refine ? (mx <= cfg.tol ? 0 : -3) : 1;
            else action = (mx <= cfg.tol) ? 0 : -3;
            ss.action = action;
        }
        prev = mx;
        wsync();
        const int action = ss.action;
        if (action != 1) {
            if (threadIdx.x == 0 && cl.rank == 0) {
                E.status[j] = action;
                E.sweeps[j] = sweeps;
            }
            break;
        }
        solve_one(Jb, l_lo, l_hi, smb, sh.rows, sh.src, &sh.cnt);
        for (int64_t idx = x_lo + threadIdx.x; idx < x_hi; idx += NT) X[idx] = X[idx] + ccast<double>(sl.x[idx]);
        ++sweeps;
    }
    wsync();
}

// KEPT: the slots hold T's values (a kernel of its own: as a branch, the other residual cost a batch 1 to 2 %)
template <typename R, bool KEPT>
__global__ void __launch_bounds__(sizeof(R) == 4 ? NT + 32 : NT, 1)
    dense_sample_kernel(const DenseNep* __restrict__ neps, const DenseSampleJob* __restrict__ jobs, int njobs,
                        int n_max, int L_max, int64_t nnz_max, unsigned char* slots, size_t slot_stride, float* img, size_t img_stride,
                        size_t img_b, int32_t* __restrict__ next, DenseSampleCfg cfg) {
    extern __shared__ __align__(16) unsigned char dense_smem[];
    cplx<R>* sm = reinterpret_cast<cplx<R>*>(dense_smem);
    __shared__ DShared sh;
    __shared__ SampleShared ss;
    __shared__ __align__(8) TcShared ts;
    TcPhase ph;
    constexpr bool tc = sizeof(R) == 4;
    cg::cluster_group cluster = cg::this_cluster();
    Cluster cl;
    cl.rank = (int)cluster.block_rank();
    cl.size = (int)cluster.num_blocks();
    cl.polls = dense_wait_polls(n_max, (L_max + cl.size - 1) / cl.size);
    if (threadIdx.x == 0) {
        mbar_init(&sh.cbar, (uint32_t)cl.size);
        sh.cabort = 0;
        ts.rank = cl.rank;
        ts.size = cl.size;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster.sync();  // the barriers exist before anyone arrives on them
    if (tc) {
        if (threadIdx.x == 0) {
            for (int i = 0; i < 7; ++i) mbar_init(&ts.bar[i], i == 3 || i == 4 ? NT / 32 : 1);
            ts.fail = 0;
            ts.stop = 0;
            ts.cmd = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (threadIdx.x < 32) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32(&ts.tmem)), "r"(TC_TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (threadIdx.x >= NT) tc_producer(dense_smem, ts);
    }
    if (threadIdx.x < NT) {
        const size_t slot = blockIdx.x / cl.size;
        const Slot<R> sl = slot_at<R>(slots + slot * slot_stride, n_max, L_max, nnz_max);
        float* my_img = img ? img + slot * img_stride : nullptr;
        for (;;) {
            // CTA 0 takes the next job for the cluster (none after a timeout)
            if (threadIdx.x == 0 && cl.rank == 0) {
                const int jb = (tc && ts.stop) || cl.fail ? njobs : atomicAdd(next, 1);
                for (int q = 0; q < cl.size; ++q) *cluster.map_shared_rank(&sh.job, q) = jb;
            }
            if (!csync(cl, sh)) break;
            const int jb = sh.job;
            if (jb >= njobs) break;
            const DenseSampleJob job = jobs[jb];
            sample_one<R, KEPT>(neps[job.nep], job.j, sl, sm, sh, ss, my_img, img_b, &ts, &ph, cfg, cl);
        }
        if (tc && threadIdx.x == 0) {
            ts.cmd = 2;
            mbar_arrive(&ts.bar[2]);
        }
    }
    if (tc) {
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (threadIdx.x < 32)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(ts.tmem), "r"(TC_TMEM_COLS)
                         : "memory");
    }
    cluster.sync();  // no CTA leaves while another may still arrive on its barrier
}

// Opt a kernel into its dynamic shared memory.  The attribute is per function and process-wide,
// so it is set to the largest allowed value rather than to this launch's size: host threads
// launching the same kernel concurrently never lower it under one another.
template <typename K>
int set_smem(K kernel, size_t bytes, const char* name) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    cudaFuncGetAttributes(&fa, kernel);
    if (bytes + fa.sharedSizeBytes > (size_t)optin)
        return set_error(RSRR_EUNSUPPORTED, std::string(name) + ": shared memory " + std::to_string(bytes) +
                                                " + " + std::to_string(fa.sharedSizeBytes) + " exceeds " +
                                                std::to_string(optin));
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         optin - (int)fa.sharedSizeBytes);
    if (e != cudaSuccess)
        return set_error(RSRR_ECUDA, std::string(name) + ": cudaFuncSetAttribute: " + cudaGetErrorString(e));
    return RSRR_OK;
}

}  // namespace

namespace {
template <typename R>
cudaLaunchConfig_t sample_config(int clusters, int cluster_size, cudaLaunchAttribute* at, cudaStream_t s) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(clusters * cluster_size));
    lc.blockDim = dim3((unsigned)(sizeof(R) == 4 ? NT + 32 : NT));
    lc.dynamicSmemBytes = std::max(factor_smem<R>(), solve_smem<R>());
    lc.stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)cluster_size;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    return lc;
}
}  // namespace

// Cluster size and count for jobs of orders n (descending): the size whose greedy schedule of the
// jobs ends first.  A point's time is taken as n^2 dense_time_share(size); no more CTAs than the largest matrix has panels, and no more clusters than there are
// slots or than the device holds at once (of 4 CTAs with 200 KB each 36 fit, of 8 CTAs 15).
template <typename R>
int dense_plan(const std::vector<int>& n, int slots, int* size, int* count) {
    RSRR_TRY(set_smem(dense_sample_kernel<R, true>, std::max(factor_smem<R>(), solve_smem<R>()), "dense_sample_kernel"));
    double best = 0.0;
    *size = 1;
    *count = 1;
    for (int c = 1; c <= kMaxCluster && (c == 1 || c * NB <= n.front()); c *= 2) {
        int fit = sm_count();
        if (c > 1) {
            cudaLaunchAttribute at[1];
            const cudaLaunchConfig_t lc = sample_config<R>(1, c, at, nullptr);
            if (cudaOccupancyMaxActiveClusters(&fit, dense_sample_kernel<R, true>, &lc) != cudaSuccess) fit = 0;
            cudaGetLastError();
            if (fit < 1) break;
        }
        const int m = std::max(1, std::min({(int)n.size(), fit, slots}));
        std::priority_queue<double, std::vector<double>, std::greater<double>> busy;
        for (int i = 0; i < m; ++i) busy.push(0.0);
        double end = 0.0;
        for (int x : n) {
            const double t = busy.top() + (double)x * x * dense_time_share(c);
            busy.pop();
            busy.push(t);
            end = std::max(end, t);
        }
        if (c == 1 || end < 0.95 * best) {
            best = end;
            *size = c;
            *count = m;
        }
    }
    return RSRR_OK;
}

template <typename R>
size_t dense_slot_bytes(int n_max, int L_max, int64_t nnz_max) {
    return slot_bytes<R>(n_max, L_max, nnz_max);
}

template <typename R>
size_t dense_image_bytes(int n_max) {
    if (sizeof(R) != 4) return 0;
    const size_t tiles = (size_t)(n_max + TC_ROWS - 1) / TC_ROWS, blocks = (size_t)(n_max + TC_COLS - 1) / TC_COLS;
    return (tiles * TC_A_FLOATS + blocks * TC_B_FLOATS) * 4;
}

template <typename R>
int launch_dense_sample(const DenseNep* d_neps, const DenseSampleJob* d_jobs, int njobs, int n_max, int L_max,
                        int64_t nnz_max, int clusters, int cluster_size, void* d_slots, void* d_img, int32_t* d_next, DenseSampleCfg cfg, cudaStream_t s) {
    if (njobs <= 0) return RSRR_OK;
    if (L_max > kMaxL) return set_error(RSRR_EINVAL, "dense sampling: L above 256");
    if (sizeof(R) == 4 && !d_img) return set_error(RSRR_EINVAL, "dense sampling: operand images missing");
    const size_t sm = std::max(factor_smem<R>(), solve_smem<R>());
    auto kernel = nnz_max > 0 ? dense_sample_kernel<R, true> : dense_sample_kernel<R, false>;
    RSRR_TRY(set_smem(kernel, sm, "dense_sample_kernel"));
    RSRR_CUDA(cudaMemsetAsync(d_next, 0, sizeof(int32_t), s));
    const size_t img_stride = dense_image_bytes<R>(n_max) / 4;
    const size_t img_b = sizeof(R) == 4 ? (size_t)((n_max + TC_ROWS - 1) / TC_ROWS) * TC_A_FLOATS : 0;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t lc = sample_config<R>(clusters, cluster_size, at, s);
    RSRR_CUDA(cudaLaunchKernelEx(&lc, kernel, d_neps, d_jobs, njobs, n_max, L_max, nnz_max,
                                 static_cast<unsigned char*>(d_slots), dense_slot_bytes<R>(n_max, L_max, nnz_max),
                                 static_cast<float*>(d_img), img_stride, img_b, d_next, cfg));
    note_launch();
    RSRR_CUDA(cudaGetLastError());
    return RSRR_OK;
}

template int dense_plan<float>(const std::vector<int>&, int, int*, int*);
template int dense_plan<double>(const std::vector<int>&, int, int*, int*);
template size_t dense_slot_bytes<float>(int, int, int64_t);
template size_t dense_slot_bytes<double>(int, int, int64_t);
template size_t dense_image_bytes<float>(int);
template size_t dense_image_bytes<double>(int);
template int launch_dense_sample<float>(const DenseNep*, const DenseSampleJob*, int, int, int, int64_t, int, int, void*, void*,
                                        int32_t*, DenseSampleCfg, cudaStream_t);
template int launch_dense_sample<double>(const DenseNep*, const DenseSampleJob*, int, int, int, int64_t, int, int, void*, void*,
                                         int32_t*, DenseSampleCfg, cudaStream_t);

}  // namespace rsrr
