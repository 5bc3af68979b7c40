// Device arithmetic of the pair loop, evaluated on arrays (test infrastructure):
// pair_weights and fast_rcp<double> exactly as the step kernels inline them.
#include "wdlb_kernels.cuh"

using namespace wdlb;

namespace {

template <int CL, class T>
__global__ void k_pair(int n, const T *in, T *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T *a = in + 6 * (size_t)i;      // s0, noff, dh+, dn+, dh-, dn-
    T qp, qm, qd;
    pair_weights<CL, T>(a[0], a[1], a[2], a[3], a[4], a[5], qp, qm, qd);
    out[3 * (size_t)i] = qp;
    out[3 * (size_t)i + 1] = qm;
    out[3 * (size_t)i + 2] = qd;
}

__global__ void k_rcp(int n, const double *in, double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fast_rcp<double>(in[i]);
}

// in: n * ni values, out: n * no values, both on the host
template <class T, class F>
int on_device(int n, int ni, int no, const T *in, T *out, F launch)
{
    T *d = nullptr;
    const size_t bi = sizeof(T) * n * ni, bo = sizeof(T) * n * no;
    if (n < 1 || cudaMalloc(&d, bi + bo) != cudaSuccess) return 1;
    T *o = d + (size_t)n * ni;
    cudaError_t e = cudaMemcpy(d, in, bi, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        launch((n + 255) / 256, d, o);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, o, bo, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 1;
}

template <class T>
int pairs(int closure, int n, const T *in, T *out)
{
    return on_device(n, 6, 3, in, out, [&](int blocks, const T *d, T *o) {
        if (closure == 0)
            k_pair<0, T><<<blocks, 256>>>(n, d, o);
        else
            k_pair<1, T><<<blocks, 256>>>(n, d, o);
    });
}

}  // namespace

extern "C" int pair_weights_f32(int closure, int n, const float *in, float *out) { return pairs(closure, n, in, out); }
extern "C" int pair_weights_f64(int closure, int n, const double *in, double *out) { return pairs(closure, n, in, out); }
extern "C" int rcp_f64(int n, const double *in, double *out)
{
    return on_device(n, 1, 1, in, out, [&](int blocks, const double *d, double *o) { k_rcp<<<blocks, 256>>>(n, d, o); });
}
