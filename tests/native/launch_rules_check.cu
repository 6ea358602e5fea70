// Host-side check of the launch rules (launch.h), no GPU needed.  Prints the
// number of checks; exits non-zero on the first failure.
#include <cstdio>
#include <cstdlib>

#include "launch.h"

namespace mpa {
std::atomic<long long> g_launches{0};
std::atomic<long long> g_fail_countdown{-1};
std::atomic<int> g_fail_code{0};
std::atomic<bool> g_prof_on{false};
}  // namespace mpa
using namespace mpa;

static int g_checked = 0;
static void expect(bool ok, const char* what) {
    ++g_checked;
    if (!ok) {
        std::printf("failed: %s\n", what);
        std::exit(1);
    }
}

int main() {
    // two blocks an SM fill it twice over, whatever the number of SMs
    for (int sms : {1, 76, 132, 148, 152, 160}) {
        expect(!fills_twice(0, sms) && !fills_twice(2ll * sms - 1, sms), "one block short");
        expect(fills_twice(2ll * sms, sms) && fills_twice(1ll << 40, sms), "filled");
    }
    std::printf("checked %d\n", g_checked);
    return 0;
}
