// The integer double arithmetic (csrc/soft64.cuh) beside the hardware's on the device, for test_soft64_device_gpu.py.
#include "physics.cuh"

namespace {

__global__ void k_mul(const double *a, const double *b, long long n, double *soft, double *hw) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    soft[i] = ck::s64_mul(a[i], b[i]);
    hw[i] = __dmul_rn(a[i], b[i]);
}
__global__ void k_float(const double *a, long long n, float *soft, float *hw, int *ok) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    bool k = true;
    soft[i] = ck::s64_to_float(a[i], k);
    hw[i] = __double2float_rn(a[i]);
    ok[i] = k;
}
template <int V, int M>
__global__ void k_accel(double R1, const double *y, long long n, double *soft, double *hw, int *ok) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double *s = y + 6 * i;
    double *u = soft + 4 * i, *v = hw + 4 * i;
    ok[i] = ck::s64_ok(ck::accel64_form<ck::MulInt, V, M>(R1, s[0], s[1], s[3], s[4], s[5], u[0], u[1], u[2], u[3]));
    ck::accel64_form<ck::MulHW, V, M>(R1, s[0], s[1], s[3], s[4], s[5], v[0], v[1], v[2], v[3]);
}
int launched() { return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1; }

}  // namespace

// all pointers: device memory; n > 0
extern "C" {
int s64d_mul(const double *a, const double *b, long long n, double *soft, double *hw) {
    k_mul<<<(unsigned)((n + 255) / 256), 256>>>(a, b, n, soft, hw);
    return launched();
}
int s64d_float(const double *a, long long n, float *soft, float *hw, int *ok) {
    k_float<<<(unsigned)((n + 255) / 256), 256>>>(a, n, soft, hw, ok);
    return launched();
}
// vm: 1 radial extraordinary, 2 azimuthal ordinary, 3 azimuthal extraordinary; soft, hw: 4 values per state
int s64d_accel(int vm, double R1, const double *y, long long n, double *soft, double *hw, int *ok) {
    const unsigned g = (unsigned)((n + 255) / 256);
    if (vm == 1) k_accel<ck::V_RADIAL, ck::M_EXT><<<g, 256>>>(R1, y, n, soft, hw, ok);
    else if (vm == 2) k_accel<ck::V_AZIMUTHAL, ck::M_ORD><<<g, 256>>>(R1, y, n, soft, hw, ok);
    else k_accel<ck::V_AZIMUTHAL, ck::M_EXT><<<g, 256>>>(R1, y, n, soft, hw, ok);
    return launched();
}
}
