// Dense FP64 complex building blocks for the projection and reduced-solve stages.
#pragma once

#include "common.cuh"

namespace rsrr {

enum { OP_N = 0, OP_T = 1, OP_C = 2 };

// C = alpha op(A) op(B) + beta C for `batch` independent problems (strided).
// op(A) is M x K, op(B) is K x N, all column-major.
struct Zgemm {
    int opA = OP_N, opB = OP_N;
    int M = 0, N = 0, K = 0;
    c128 alpha{1, 0}, beta{0, 0};
    const c128* A = nullptr;
    int64_t lda = 0, sA = 0;
    const c128* B = nullptr;
    int64_t ldb = 0, sB = 0;
    c128* C = nullptr;
    int64_t ldc = 0, sC = 0;
    int batch = 1;
    bool fp64 = false;  // FP64 CUDA cores whatever the path: products whose terms must keep their own scale
};
int zgemm(const Zgemm& g, cudaStream_t s);
// In-place inverses of `batch` dense k x k complex128 matrices (column-major, stride k^2) by
// blocked Gauss-Jordan elimination with partial pivoting (zinv.cu); info[t] (zeroed by the
// caller) is set to 1 where matrix t met an exactly zero pivot column.  zinv_block(k) is the block
// width, 0 when a k-row panel does not fit shared memory (EUNSUPPORTED).
int zinv_block(int k);
size_t zinv_bytes_per_matrix(int k);
int zinv_batch(c128* X, int k, int batch, int32_t* info, cudaStream_t st);
// FP64-accurate ZGEMM on the tensor cores (exact BF16 digit products, see zgemm_tc.cu), and
// the shapes for which zgemm() takes it.  zgemm_path: 0 = by shape, 1 = FP64 CUDA cores only,
// 2 = tensor cores for every shape (per host thread; for tests and measurements).
int zgemm_tc(const Zgemm& g, cudaStream_t s);
// While one is alive (and begin() succeeded), the tensor-core ZGEMMs of this host thread do not wait
// for their kernel: a bounded wait that gave up is recorded in one device word, which check() reads
// after synchronising `st`.  The products must all run on `st`.  check() ends the deferral.  A call that
// fails before its check() passes its status through failed(): what it met may be a product that was
// never written, so a recorded timeout takes the status's place.
class ZgemmDefer {
  public:
    explicit ZgemmDefer(cudaStream_t s) : st(s) {}
    ~ZgemmDefer();
    ZgemmDefer(const ZgemmDefer&) = delete;
    ZgemmDefer& operator=(const ZgemmDefer&) = delete;
    int begin();
    int check();
    int failed(int rc);
    int* device_word() const { return word; }

  private:
    cudaStream_t st;
    int* word = nullptr;
    int* outer = nullptr;  // the deferral that was in force before this one
    bool on = false;
};
// Suspends the deferral while user code runs on this host thread: products that a callback asks for have
// their own stream and wait for themselves.
class ZgemmNoDefer {
  public:
    ZgemmNoDefer();
    ~ZgemmNoDefer();
    ZgemmNoDefer(const ZgemmNoDefer&) = delete;
    ZgemmNoDefer& operator=(const ZgemmNoDefer&) = delete;

  private:
    int* outer;
};
bool zgemm_tc_fits(const Zgemm& g);
void zgemm_set_path(int path);
int zgemm_get_path();
// Accounting of the ZGEMMs issued by this host thread between the two calls.
void zgemm_profile_begin();
void zgemm_profile_end(double* ms, double* flops, double* ms_tc = nullptr, double* flops_tc = nullptr);
// Accounting of the one-sided Jacobi sweeps (device time of the sweep kernels, algorithmic flops).
void jacobi_profile_begin();
void jacobi_profile_end(double* ms, double* flops);
// One-sided Jacobi SVD of a square D x D matrix with a QR preconditioner (project.cu): on return H
// holds U Sigma and Jr the right singular vectors, as jacobi_orthogonalize(H, ..., Jr) would give.
int jacobi_svd_preconditioned(c128* H, int D, c128* Jr, cudaStream_t st, double floor, double conv, int* sweeps);

// Sum of v over a CTA (blockDim a multiple of 32, <= 1024); every thread gets the result.
// Four block-wide sums at once (two CTA barriers instead of eight); every thread gets them.
__device__ __forceinline__ void block_sum4(double& a, double& b, double& c, double& d) {
    __shared__ double red4_[4][33];
    for (int off = 16; off; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
        c += __shfl_down_sync(0xffffffffu, c, off);
        d += __shfl_down_sync(0xffffffffu, d, off);
    }
    __syncthreads();
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) { red4_[0][w] = a; red4_[1][w] = b; red4_[2][w] = c; red4_[3][w] = d; }
    __syncthreads();
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = 0; i < nw; ++i)
        for (int j = 0; j < 4; ++j) s[j] += red4_[j][i];
    a = s[0];
    b = s[1];
    c = s[2];
    d = s[3];
}

__device__ __forceinline__ double block_sum_all(double v) {
    __shared__ double red_[33];
    for (int off = 16; off; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red_[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double r = (threadIdx.x < (blockDim.x >> 5)) ? red_[threadIdx.x] : 0.0;
        for (int off = 16; off; off >>= 1) r += __shfl_down_sync(0xffffffffu, r, off);
        if (threadIdx.x == 0) red_[32] = r;
    }
    __syncthreads();
    return red_[32];
}

// Device-wide barrier for cooperative kernels.  Every wait is bounded: after the spin limit
// the barrier records a timeout in *err and returns false, and the kernel returns.
// One word: every CTA adds 1 but CTA 0, which adds 2^31 - (n - 1), so the top bit flips when all n
// have arrived and the low bits are zero again.  A CTA reads the top bit when the kernel starts (it
// cannot flip before that CTA's own arrival) and then polls the word it added to: one trip to L2
// and back, 1.27 us with 152 CTAs, against 2.31 us for an arrival count whose last CTA releases
// the others through a second word.
struct GridBar {
    unsigned* count;
    int* err;
    long long spin_limit;  // polls of about half a microsecond before a wait gives up
    unsigned ctas;         // 0: gridDim.x
};
// The two words sit on separate 128-byte lines.
constexpr int kGridBarWords = 64;  // allocation size in unsigned words
constexpr int kGridBarErrWord = 32;
inline GridBar grid_bar_at(unsigned* base, long long spin_limit = 1LL << 22, unsigned ctas = 0) {
    return GridBar{base, reinterpret_cast<int*>(base + kGridBarErrWord), spin_limit, ctas};
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu(unsigned* p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// The barrier's phase, read once at the start of the kernel (meaningful in thread 0).
__device__ __forceinline__ unsigned grid_phase(const GridBar& gb) {
    return threadIdx.x == 0 ? ld_acquire_gpu(gb.count) & 0x80000000u : 0u;
}
__device__ __forceinline__ bool grid_sync(const GridBar& gb, unsigned& phase) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned n = gb.ctas ? gb.ctas : gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(gb.count),
                     "r"(blockIdx.x == 0 ? 0x80000000u - (n - 1) : 1u) : "memory");
        int ok = 1;
        long long spins = 0;
        while (((ld_acquire_gpu(gb.count) ^ phase) & 0x80000000u) == 0) {
            // bounded: give up, report, return; also when another CTA has
            if (++spins > gb.spin_limit || ((spins & 255) == 0 && *(volatile int*)gb.err != 0)) {
                atomicExch(gb.err, 1);
                ok = 0;
                break;
            }
        }
        phase ^= 0x80000000u;
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}


// One-sided (Hestenes) Jacobi on the k columns of B (mb x k, ld mb), accumulating the
// rotations into J (k x k, ld k, initialised to I by the caller when wanted; may be null).
// Sweeps stop once every pair of columns above abs_floor has |<b_p, b_q>| / (|b_p| |b_q|) <=
// conv (singular values are then exact to second order in conv); columns below abs_floor are
// not rotated.
int jacobi_orthogonalize(c128* B, int mb, int k, c128* J, cudaStream_t s, int max_sweeps, int* sweeps_out,
                         double abs_floor, double conv);

// Column 2-norms of B (mb x k) into out[k] (device).
void column_norms(const c128* B, int mb, int k, int64_t ld, double* out, cudaStream_t s);

// Frobenius norm squared of the block rows [r0, r1) x cols [c0, c1) of A (ld lda), added
// atomically to *out (device, caller zeroes it).
void block_norm2(const c128* A, int64_t lda, int r0, int r1, int c0, int c1, double* out, cudaStream_t s);

}  // namespace rsrr
