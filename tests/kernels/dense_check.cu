// The sweep's tensor-core contractions on their own, for tests/test_gpu_dense.py:
// C = op(A) B (tc_dense) and the rank-b update W -= C X of the inverse (tc::zupdate),
// in double-float and binary64.  One block; device pointers; returns the kernel's
// time-out flag, or -1 for a CUDA error.
#include "rgf_steps.cuh"

using namespace rgf;

namespace {

constexpr int kSmem = 200 * 1024;
constexpr int kTcBytes = (int)((tc::smem_bytes() + 1023) / 1024 * 1024);

template <class R>
__global__ void __launch_bounds__(NT, 1)
product(int m, int n, int k, const cx<R>* A, int lda, const cx<R>* B, int ldb, cx<R>* C, int ldc, bool ta, int* err) {
    const tc::Area ar{0};
    const uint32_t phase = tc::setup(ar);
    tc_dense<R>(m, n, k, A, lda, B, ldb, C, ldc, ta, ar, phase);
    if (threadIdx.x == 0) *err = *(volatile int*)ar.err();
    tc::teardown(ar);
}

template <class R>
__global__ void __launch_bounds__(NT, 1)
update(int K, int bb, const cx<R>* C, const cx<R>* X, cx<R>* W, int r0, int M, int j0, int N, int* err) {
    const tc::Area ar{0};
    const uint32_t phase = tc::setup(ar);
    cx<R>* Cs = reinterpret_cast<cx<R>*>(rgf_dyn_smem + kTcBytes);
    cx<R>* Xs = Cs + bb * K;
    for (int e = threadIdx.x; e < bb * K; e += NT) {
        Cs[e] = C[e];
        Xs[e] = X[e];
    }
    __syncthreads();
    tc::zupdate<cx<R>>(tc::dyn_off(Cs), tc::dyn_off(Xs), K, bb, W, K, r0, M, j0, N, ar, phase);
    if (threadIdx.x == 0) *err = *(volatile int*)ar.err();
    tc::teardown(ar);
}

template <class F, class... Args>
int run(F kern, Args... args) {
    int *err = nullptr, h = -1;
    if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) return -1;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e == cudaSuccess) {
        kern<<<1, NT, kSmem>>>(args..., err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h, err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(err);
    return e == cudaSuccess ? h : -1;
}

}  // namespace

extern "C" int check_product(int f64, int ta, int m, int n, int k, const void* A, int lda, const void* B, int ldb,
                             void* C, int ldc) {
    if (m < 1 || n < 1 || k < 1 || lda < (ta ? m : k) || ldb < n || ldc < n) return -1;
    return f64 ? run(product<double>, m, n, k, (const zd*)A, lda, (const zd*)B, ldb, (zd*)C, ldc, ta != 0)
               : run(product<df32>, m, n, k, (const zf*)A, lda, (const zf*)B, ldb, (zf*)C, ldc, ta != 0);
}

// C, X [bb][K], W [K columns][K]; columns l outside the panel j0 .. j0 + bb - 1, N of them.
extern "C" int check_update(int f64, int K, int bb, const void* C, const void* X, void* W, int r0, int M, int j0, int N) {
    if (bb < 1 || bb > 16 || M < 1 || M > 128 || r0 < 0 || r0 + M > K || j0 < 0 || N < 1 || N + bb > K || j0 + bb > K ||
        kTcBytes + 2 * K * bb * 16 > kSmem)
        return -1;
    return f64 ? run(update<double>, K, bb, (const zd*)C, (const zd*)X, (zd*)W, r0, M, j0, N)
               : run(update<df32>, K, bb, (const zf*)C, (const zf*)X, (zf*)W, r0, M, j0, N);
}
