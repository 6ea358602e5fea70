// What launch_pdl leaves behind when the runtime refuses a launch for its grid
// (more than 65535 blocks in y; nothing runs): the error is returned and is not
// found again by the next check of the runtime's last error.
#include <cstdio>

#include "launch.h"

namespace mpa {
std::atomic<long long> g_launches{0};
std::atomic<long long> g_fail_countdown{-1};
std::atomic<int> g_fail_code{0};
std::atomic<bool> g_prof_on{false};
}  // namespace mpa

__global__ void nothing_kernel(int) {}

int main() {
    for (bool early : {false, true}) {
        const cudaError_t e = mpa::launch_pdl(early, nothing_kernel, dim3(1, 70000), 32, 0, nullptr, 0);
        const cudaError_t left = cudaPeekAtLastError();
        std::printf("returned %d, left %d\n", (int)e, (int)left);
        if (e != cudaErrorInvalidConfiguration && e != cudaErrorInvalidValue) return 2;
        if (left != cudaSuccess) return 1;
    }
    return 0;
}
