// Batched in-place inverse of dense complex128 matrices by blocked Gauss-Jordan elimination with
// partial pivoting: the N_S inverses T_S(z_j)^{-1} of the reduced solve (Algorithm 1, the moments
// of Eq. eq-Ap-num need the whole inverse at every quadrature point).
//
// Per block column J = [jb, jb + bb) of the in-place matrix M (k x k, column-major):
//   1. panel (CUDA cores, one CTA per matrix): LU with partial pivoting (cabs1, lowest row on
//      ties) of a copy of rows jb..k-1 of the block column, in shared memory; it picks the bb
//      pivot rows, which are swapped into rows J across the whole matrix.  With D = M_JJ after
//      the swaps (its LU is the top of the panel), D^{-1} = U11^{-1} L11^{-1}.
//      E = M_:J with rows J cleared is kept, then M_:J is set to [0; I].
//   2. W = D^{-1} M_J: (bb x k, one batched ZGEMM), copied into rows J of M.
//   3. trailing update (one batched ZGEMM over all matrices, K = bb):  M -= E W.
//      Rows J are left as W (E is zero there); the other rows get M_O: - M_OJ D^{-1} M_J:, and
//      the pivot columns become -M_OJ D^{-1} (rows O) and D^{-1} (rows J): the Gauss-Jordan step.
// After the last block the row interchanges, applied to whole rows throughout, are undone on the
// columns in reverse order: inv(A) = inv(P A) P.
//
// The elimination costs k^3 complex multiply-adds per matrix, as LU plus an inverse from the
// factors does; nearly all of it is in the ZGEMMs (k x k x bb each), which take the FP64-accurate
// tensor-core emulation when the batch is large enough.  The panels are FP64 CUDA-core work, k bb / 2
// multiply-adds a column, at two a clock per SM: every instruction that a warp repeats for nothing
// counts there, so reciprocals are taken once a column by one warp, D^{-1} comes from block-wise
// triangular inverses and W is a batched product whose tiles fill the SMs evenly.  The nine
// panels of 500 matrices with k = 280 took 30.7 ms with the reciprocal in every thread, D^{-1} by columns
// and W by the matrix's own CTA; now 8.7 ms, and W's products 9.7 ms (8.3 at the FP64 rate).
#include <algorithm>

#include "dense.cuh"

namespace rsrr {

namespace {

constexpr int kZiThreads = 512;
constexpr int kZiWarps = kZiThreads / 32;
constexpr unsigned FULLM = 0xffffffffu;
constexpr size_t kZiSmemMax = 225 * 1024;

// The two triangular inverses take the panel's place once it has been used, so they cost no block
// width: 32 columns up to k = 450 (with a place of their own up to 384: at k = 404, 500 matrices,
// 16-column blocks took 156 ms, 32-column ones take 105).
size_t panel_smem(int rows, int bb) {
    return std::max((size_t)rows * bb, (size_t)2 * 32 * 33) * sizeof(c128);
}

__global__ void __launch_bounds__(kZiThreads) zinv_panel_kernel(c128* X, int k, int jb, int bb, int b, int32_t* piv,
                                                               c128* E, c128* Dv, int32_t* info) {
    extern __shared__ __align__(16) unsigned char zi_raw[];
    __shared__ double s_best[kZiWarps];
    __shared__ int s_pos[kZiWarps];
    __shared__ int s_piv[32];
    __shared__ int s_sing;
    __shared__ c128 s_inv[32];  // 1 / pivot
    const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t kk = (int64_t)k * k;
    c128* Xm = X + (int64_t)t * kk;
    c128* Et = E + (int64_t)t * k * b;
    c128* Dt = Dv + (int64_t)t * b * b;
    const int rows = k - jb;
    c128* P = reinterpret_cast<c128*>(zi_raw);  // [bb][rows], column-major
    c128* Ui = P;             // [32][33] U11^{-1}, column-major, over the panel
    c128* Li = Ui + 32 * 33;  // [32][33] L11^{-1}
    if (tid == 0) s_sing = 0;
    for (int idx = tid; idx < rows * bb; idx += kZiThreads) {
        const int r = idx % rows, c = idx / rows;
        P[idx] = Xm[(int64_t)(jb + r) + (int64_t)(jb + c) * k];
    }
    __syncthreads();

    // ---- LU with partial pivoting of the panel copy ------------------------------------------
    for (int i = 0; i < bb; ++i) {
        double best = -1.0;
        int pos = rows;
        for (int r = i + tid; r < rows; r += kZiThreads) {
            const double a = cabs1(P[r + (int64_t)i * rows]);
            if (a > best) { best = a; pos = r; }
        }
        for (int off = 16; off; off >>= 1) {
            const double ob = __shfl_down_sync(FULLM, best, off);
            const int op = __shfl_down_sync(FULLM, pos, off);
            if (ob > best || (ob == best && op < pos)) { best = ob; pos = op; }
        }
        if (lane == 0) { s_best[warp] = best; s_pos[warp] = pos; }
        __syncthreads();
        if (warp == 0) {
            best = lane < kZiWarps ? s_best[lane] : -1.0;
            pos = lane < kZiWarps ? s_pos[lane] : rows;
            for (int off = 16; off; off >>= 1) {
                const double ob = __shfl_down_sync(FULLM, best, off);
                const int op = __shfl_down_sync(FULLM, pos, off);
                if (ob > best || (ob == best && op < pos)) { best = ob; pos = op; }
            }
            if (lane == 0) {
                // an exactly zero (or non-finite) column: singular; keep going with the diagonal
                // entry so that the launch stays well defined, the caller reports the point
                if (!(best > 0.0) || pos >= rows) { s_sing = 1; pos = i; }
                s_piv[i] = pos;
                const c128 d = P[pos + (int64_t)i * rows];
                s_inv[i] = cis_zero(d) ? mk<double>(1.0, 0.0) : crecip(d);
            }
        }
        __syncthreads();
        const int p = s_piv[i];
        if (p != i && tid < bb) {
            const c128 tmp = P[i + (int64_t)tid * rows];
            P[i + (int64_t)tid * rows] = P[p + (int64_t)tid * rows];
            P[p + (int64_t)tid * rows] = tmp;
        }
        __syncthreads();
        const c128 dinv = s_inv[i];
        for (int r = i + 1 + tid; r < rows; r += kZiThreads) P[r + (int64_t)i * rows] = P[r + (int64_t)i * rows] * dinv;
        __syncthreads();
        const int nr = rows - i - 1, nc = bb - i - 1;
        for (int idx = tid; idx < nr * nc; idx += kZiThreads) {
            const int r = i + 1 + idx % nr, c = i + 1 + idx / nr;
            cfms(P[r + (int64_t)c * rows], P[r + (int64_t)i * rows], P[i + (int64_t)c * rows]);
        }
        __syncthreads();
    }

    // ---- the interchanges on whole rows of M, the kept block column E, M_:J = [0; I] -----------
    if (tid < bb) piv[(int64_t)t * k + jb + tid] = jb + s_piv[tid];
    for (int c = tid; c < k; c += kZiThreads) {
        c128* col = Xm + (int64_t)c * k + jb;
        for (int i = 0; i < bb; ++i) {
            const int p = s_piv[i];
            if (p != i) {
                const c128 tmp = col[i];
                col[i] = col[p];
                col[p] = tmp;
            }
        }
    }
    __syncthreads();
    for (int idx = tid; idx < k * bb; idx += kZiThreads) {
        const int r = idx % k, c = idx / k;
        c128* xp = Xm + r + (int64_t)(jb + c) * k;
        Et[r + (int64_t)c * k] = (r >= jb && r < jb + bb) ? czero<double>() : *xp;
        *xp = (r == jb + c) ? mk<double>(1.0, 0.0) : czero<double>();
    }

    // ---- D^{-1} = U11^{-1} L11^{-1} ------------------------------------------------------------
    // Both triangular inverses grow from blocks of one column: [A, B; 0, C]^{-1} has -A^{-1} B C^{-1}
    // off the diagonal (and its mirror image for L).  At level w there are 16 w such entries a factor;
    // threads 0..255 take U's, threads 256..511 L's.
    constexpr int kTri = 32 * 32 / kZiThreads;
    c128 tri[kTri];
#pragma unroll
    for (int q = 0; q < kTri; ++q) {
        const int idx = tid + q * kZiThreads, r = idx % 32, c = idx / 32;
        tri[q] = r < bb && c < bb ? P[r + (int64_t)c * rows] : czero<double>();
    }
    __syncthreads();  // the panel has been read
#pragma unroll
    for (int q = 0; q < kTri; ++q) {
        const int idx = tid + q * kZiThreads, r = idx % 32, c = idx / 32;
        const bool in = r < bb && c < bb;
        const c128 v = tri[q];
        Ui[r + 33 * c] = r == c ? (in ? s_inv[c] : czero<double>()) : r < c ? v : czero<double>();
        Li[r + 33 * c] = r == c ? mk<double>(in ? 1.0 : 0.0, 0.0) : r > c ? v : czero<double>();
    }
    __syncthreads();
    {
        const int h = tid >> 8, e = tid & 255;
        c128* T = h ? Li : Ui;
        // entry (x, y) of the upper factor, (y, x) of the lower one: the same formulas for both with the
        // order of the products exchanged
        auto at = [&](int x, int y) -> c128& { return h ? T[y + 33 * x] : T[x + 33 * y]; };
        for (int w = 1; w < 32; w *= 2) {
            const int b0 = 2 * w * (e / (w * w)), x = b0 + e % w, y = b0 + w + (e % (w * w)) / w;
            const bool on = e < 16 * w && y < bb;
            c128 v = czero<double>();
            if (on)
                for (int l = x; l < b0 + w; ++l) cfma(v, at(x, l), at(l, y));  // A^{-1} B
            __syncthreads();
            if (on) at(x, y) = v;
            __syncthreads();
            v = czero<double>();
            if (on)
                for (int l = b0 + w; l <= y; ++l) cfms(v, at(x, l), at(l, y));  // -(A^{-1} B) C^{-1}
            __syncthreads();
            if (on) at(x, y) = v;
            __syncthreads();
        }
    }
    for (int idx = tid; idx < bb * bb; idx += kZiThreads) {
        const int r = idx % bb, c = idx / bb;
        c128 v = czero<double>();
        for (int l = max(r, c); l < bb; ++l) cfma(v, Ui[r + 33 * l], Li[l + 33 * c]);
        Dt[r + (int64_t)c * b] = v;
    }
    if (tid == 0 && s_sing) info[t] = 1;
}

// rows jb .. jb + bb - 1 of every matrix <- W
__global__ void zinv_rows_kernel(c128* X, int k, int jb, int bb, int b, const c128* Wb) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)bb * k) return;
    const int i = (int)(idx % bb), c = (int)(idx / bb), t = blockIdx.y;
    X[(int64_t)t * k * k + jb + i + (int64_t)c * k] = Wb[(int64_t)t * b * k + i + (int64_t)c * b];
}

// inv(A) = inv(P A) P: the interchanges of rows i <-> piv[i], undone on the columns from the last.
__global__ void zinv_unpermute_kernel(c128* X, int k, const int32_t* piv) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.y;
    if (r >= k) return;
    c128* Xm = X + (int64_t)t * k * k;
    const int32_t* pv = piv + (int64_t)t * k;
    for (int i = k - 1; i >= 0; --i) {
        const int p = pv[i];
        if (p != i) {
            const c128 tmp = Xm[r + (int64_t)i * k];
            Xm[r + (int64_t)i * k] = Xm[r + (int64_t)p * k];
            Xm[r + (int64_t)p * k] = tmp;
        }
    }
}

}  // namespace

int zinv_block(int k) {
    for (int b : {32, 16, 8})
        if (panel_smem(k, std::min(b, k)) <= kZiSmemMax) return b;
    return 0;
}

size_t zinv_bytes_per_matrix(int k) {
    const int b = std::max(1, zinv_block(k));
    // M, E, W, D^{-1}, pivots, and the emulated ZGEMM's digit images of E and W (about 3 KB per row)
    return (size_t)k * k * sizeof(c128) + (size_t)(2 * k + b) * b * sizeof(c128) + (size_t)k * 4 + (size_t)3072 * k + 256;
}

int zinv_batch(c128* X, int k, int batch, int32_t* info, cudaStream_t st) {
    const int b = zinv_block(k);
    if (b == 0) return set_error(RSRR_EUNSUPPORTED, "zinv_batch: matrix too large for shared-memory panels");
    if (k < 1 || batch < 1) return set_error(RSRR_EINVAL, "zinv_batch: empty problem");
    c128 *E = nullptr, *Wb = nullptr, *Dv = nullptr;
    int32_t* piv = nullptr;
    auto release = [&]() {
        dfree(E, st);
        dfree(Wb, st);
        dfree(Dv, st);
        dfree(piv, st);
    };
    int rc = RSRR_OK;
    if ((rc = dalloc_n(&E, (size_t)batch * k * b, st)) || (rc = dalloc_n(&Wb, (size_t)batch * b * k, st)) ||
        (rc = dalloc_n(&Dv, (size_t)batch * b * b, st)) || (rc = dalloc_n(&piv, (size_t)batch * k, st))) {
        release();
        return rc;
    }
    static bool attr_set = false;  // the same value every time
    if (!attr_set) {
        cudaFuncSetAttribute(zinv_panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kZiSmemMax);
        attr_set = true;
    }
    for (int jb = 0; jb < k && rc == RSRR_OK; jb += b) {
        const int bb = std::min(b, k - jb);
        { zinv_panel_kernel<<<batch, kZiThreads, panel_smem(k - jb, bb), st>>>(X, k, jb, bb, b, piv, E, Dv, info); note_launch(); }
        if (cudaGetLastError() != cudaSuccess) {
            rc = set_error(RSRR_ECUDA, "zinv_panel_kernel launch");
            break;
        }
        Zgemm gw;  // W = D^{-1} M_J: (rows J hold the swapped pivot rows, their J columns the identity)
        gw.opA = OP_N; gw.opB = OP_N; gw.M = bb; gw.N = k; gw.K = bb;
        gw.A = Dv; gw.lda = b; gw.sA = (int64_t)b * b;
        gw.B = X + jb; gw.ldb = k; gw.sB = (int64_t)k * k;
        gw.C = Wb; gw.ldc = b; gw.sC = (int64_t)b * k;
        gw.batch = batch;
        // FP64 cores: the emulation's error is normwise in each row of D^{-1} and column of M_J, and on
        // matrices with graded rows (8 decades) that loses 5 digits of the inverse
        gw.fp64 = true;
        if ((rc = zgemm(gw, st)) != RSRR_OK) break;
        { zinv_rows_kernel<<<dim3((unsigned)ceil_div((int64_t)bb * k, 256), (unsigned)batch), 256, 0, st>>>(X, k, jb, bb, b, Wb); note_launch(); }
        Zgemm g;
        g.opA = OP_N; g.opB = OP_N; g.M = k; g.N = k; g.K = bb;
        g.alpha = mk<double>(-1.0, 0.0);
        g.beta = mk<double>(1.0, 0.0);
        g.A = E; g.lda = k; g.sA = (int64_t)k * b;
        g.B = Wb; g.ldb = b; g.sB = (int64_t)b * k;
        g.C = X; g.ldc = k; g.sC = (int64_t)k * k;
        g.batch = batch;
        rc = zgemm(g, st);
    }
    if (rc == RSRR_OK) {
        dim3 g((unsigned)ceil_div(k, 256), (unsigned)batch);
        { zinv_unpermute_kernel<<<g, 256, 0, st>>>(X, k, piv); note_launch(); }
        if (cudaGetLastError() != cudaSuccess) rc = set_error(RSRR_ECUDA, "zinv_unpermute_kernel launch");
    }
    release();
    return rc;
}

}  // namespace rsrr
