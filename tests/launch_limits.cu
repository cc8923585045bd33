// The launches of the compiled FFT passes on a pretended runtime: two devices with
// their own limits on the dynamic shared memory of each kernel (48 KB until raised), as
// the CUDA runtime keeps them.  Nothing runs on a GPU.  Prints one line per
// launch that its device would refuse, and per limit that a launch lowered; exits
// with the number of lines.
#include <cuda_runtime.h>

#include <cstdio>
#include <map>
#include <utility>

namespace fake {
int device = 0, faults = 0;
const char *what = "";
std::map<std::pair<int, const void *>, int> limits;
int limit(const void *k) {
    auto it = limits.find({device, k});
    return it == limits.end() ? 48 * 1024 : it->second;
}
template <class K> cudaError_t set_attribute(K *kern, cudaFuncAttribute attr, int value) {
    const void *k = reinterpret_cast<const void *>(kern);
    if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        if (value < limit(k)) std::printf("%s: device %d: limit lowered from %d to %d\n", what, device, limit(k), value), ++faults;
        limits[{device, k}] = value;
    }
    return cudaSuccess;
}
template <class K> cudaError_t occupancy(int *n, K *kern, int, size_t smem) {
    if ((int)smem > limit(reinterpret_cast<const void *>(kern))) return cudaErrorInvalidValue;
    *n = (int)(227 * 1024 / (smem + 1024));
    return cudaSuccess;
}
template <class K, class... A> cudaError_t launch(const cudaLaunchConfig_t *cfg, K *kern, A &&...) {
    const int l = limit(reinterpret_cast<const void *>(kern));
    if ((int)cfg->dynamicSmemBytes > l)
        std::printf("%s: device %d: launch with %d bytes, limit %d\n", what, device, (int)cfg->dynamicSmemBytes, l), ++faults;
    return cudaSuccess;
}
}  // namespace fake
#define cudaFuncSetAttribute fake::set_attribute
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake::occupancy
#define cudaLaunchKernelEx fake::launch
#include "fft.cuh"

template <class T, class P> void pass(const char *what, unsigned outer, int inner) {
    fake::what = what;
    mbd::FFTArgs<T> a{};
    a.K = P::K;
    a.inner = inner;
    a.V = 2;
    a.W = 32;
    a.sms = 152;
    if (mbd::ct_size<T, P>(a, 0, outer, nullptr) != 1) std::printf("%s: device %d: not launched\n", what, fake::device), ++fake::faults;
}

int main() {
    for (fake::device = 0; fake::device < 2; ++fake::device) {
        pass<float, mbd::Plan<4, 5, 10>>("200, resident tiles", 4, 64);
        pass<float, mbd::Plan<4, 5, 10>>("200, persistent blocks", 200, 6400);
        pass<float, mbd::Plan<4, 5, 10>>("200, resident tiles again", 4, 64);
        pass<double, mbd::Plan<16, 16>>("256 in double, persistent blocks", 200, 6400);
    }
    return fake::faults;
}
