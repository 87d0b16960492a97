// Device functions of the pair arithmetics evaluated over arrays, for the tests.
#include "pairkern.cuh"

using namespace ctr;

namespace {

__global__ void eval_kernel(int which, int64_t n, const double* __restrict__ x, pk::PairConsts kc, double* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (which == 0) {
        const pk::F2 e = pk::exp_neg_ffl(pk::f2(pk::split_ff_dev(x[i])), kc.exp_tab);
        out[i] = (double)e.hi + (double)e.lo;
    } else {
        out[i] = which == 1 ? pk::exp_neg_d(x[i], kc, kc.exp_tab) : pk::rsqrt_d(x[i]);
    }
}

}  // namespace

// which 0: exp_neg_ffl(x), 1: exp_neg_d(x) = e^{-kappa x}, 2: rsqrt_d(x); host arrays of n
extern "C" int eval_primitive(int which, int64_t n, const double* x, double kappa, double* out) {
    ctr_ibim s;
    s.kappa = kappa;
    s.eps_in = s.eps_out = 1.0;
    if (cudaGetDevice(&s.device) != cudaSuccess) return -1;
    pk::PairConsts kc;
    if (pair_consts(&s, which == 0 ? 1 : 2, &kc) < 0) return -2;
    DevBuf dx, dy;
    if (dx.alloc(sizeof(double) * n) < 0 || dy.alloc(sizeof(double) * n) < 0) return -3;
    if (cudaMemcpy(dx.p, x, sizeof(double) * n, cudaMemcpyHostToDevice) != cudaSuccess) return -4;
    eval_kernel<<<grid_for(n, 256), 256>>>(which, n, dx.as<double>(), kc, dy.as<double>());
    return cudaMemcpy(out, dy.p, sizeof(double) * n, cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : -5;
}
