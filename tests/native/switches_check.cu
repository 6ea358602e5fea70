// Kernels that use the switched operations of device.cuh, compiled with each
// switch away from its default.
#include "adjoint.cuh"
#include "kcs.cuh"

namespace mpa {
template __global__ void scan_pair_kernel<true>(const ScanParams<float>);
template __global__ void kc_kernel<float, 256, KC_MPA_POST>(const KCParams<float>);
template __global__ void kcs_kernel<256, KC_MPA_PRE>(const KCParams<float>);
template __global__ void kn_kernel<float, 256, true, true>(const KNParams<float>);
template __global__ void ssc_kernel<float, 64, SS_REV, 1>(const SSCParams<float>);
}  // namespace mpa
