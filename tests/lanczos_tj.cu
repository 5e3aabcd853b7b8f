// Device scalars of the Lanczos loop behind a C interface for
// test_gpu_lanczos_tj.py: rcp_f64, rsqrt_f64 and the T_j block of the update.
#include "lanczos_tj.cuh"

using namespace pse;

__global__ void k_scalars(int n, const double *x, double *rcp, double *rsq) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    rcp[i] = rcp_f64(x[i]);
    rsq[i] = rsqrt_f64(x[i]);
}

// One step of the loop: alpha_k of the k-th matrix, then its T_k block.
__global__ void k_tj(LzState *lz, int k, LzStop st, double *qlws) {
    __shared__ EigSmem sm;
    EigIn in;
    in.fetch(lz, threadIdx.x);
    lz_eig_body(lz, k, st, &sm, qlws, in);
}

template <typename T> struct Buf {
    T *p = nullptr;
    explicit Buf(size_t n) { if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess) p = nullptr; }
    ~Buf() { cudaFree(p); }
};

extern "C" int scalars_f64(int n, const double *x, double *rcp, double *rsq) {
    Buf<double> dx(n), dr(n), dq(n);
    if (!dx.p || !dr.p || !dq.p || n < 1) return 1;
    cudaMemcpy(dx.p, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    k_scalars<<<(n + 255) / 256, 256>>>(n, dx.p, dr.p, dq.p);
    cudaMemcpy(rcp, dr.p, sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(rsq, dq.p, sizeof(double) * n, cudaMemcpyDeviceToHost);
    return (int)cudaGetLastError();
}

// y[k - 1][0..k-1] = T_k^{1/2} e_1 for k = 1..K (rows of K), change[k - 1] =
// ||y_k - y_{k-1}|| / ||y_k||, stop[k - 1] the stop rule's answer.  beta_k and
// later are NaN while T_k is worked on.
extern "C" int tj_sqrt_e1(int K, const double *alpha, const double *beta, int max_iter, int fixed_iter, double tol,
                          double *y, double *change, int *stop) {
    Buf<LzState> lz(1);
    Buf<double> ws(PSE_QL_WORK);
    if (!lz.p || !ws.p || K < 1 || K > PSE_MAXIT) return 1;
    LzState h{};
    for (int i = 0; i < PSE_MAXIT + 2; ++i) h.beta[i] = nan("");
    h.beta[0] = 1.0;
    const LzStop st{max_iter, fixed_iter, tol, 0};
    for (int k = 1; k <= K; ++k) {
        h.alpha[k] = alpha[k - 1];
        if (k > 1) h.beta[k - 1] = beta[k - 2];
        cudaMemcpy(lz.p, &h, sizeof(h), cudaMemcpyHostToDevice);
        k_tj<<<1, 32>>>(lz.p, k, st, ws.p);
        cudaMemcpy(&h, lz.p, sizeof(h), cudaMemcpyDeviceToHost);
        for (int i = 0; i < k; ++i) y[(k - 1) * K + i] = h.y[i];
        change[k - 1] = h.den > 0.0 ? sqrt(h.num / h.den) : 1.0;
        stop[k - 1] = h.stop_y;
    }
    return (int)cudaGetLastError();
}
