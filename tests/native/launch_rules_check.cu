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
    // FP64 passes: CTAs that an early start would pack in pairs onto a part of
    // the SMs start after the kernel before them, all others early
    expect(pair_fits(227 * 1024 / 2 - 1024) && !pair_fits(114 * 1024), "two CTAs an SM");
    for (int sms : {132, 148, 152}) {
        for (long long b = 1; b <= 3 * sms; ++b) {
            expect(pdl_level64(false, b, sms), "one CTA an SM: early");
            expect(pdl_level64(true, b, sms) == (b <= sms / 4 || b > sms), "packed grids: ordinary");
        }
    }
    for (int l = 8; l <= 24; ++l) {
        const long long n = 1ll << l;
        expect(pdl_field<float>(n) && pdl_field<float>(n, true), "FP32 fields: early");
        expect(pdl_field<double>(n) == (l <= 15 || l > 18), "FP64 split steps");
        expect(pdl_field<double>(n, true) == (l <= 15 || l > 19), "FP64 transforms");
    }
    std::printf("checked %d\n", g_checked);
    return 0;
}
