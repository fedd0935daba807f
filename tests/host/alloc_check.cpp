// Host-side check of a buffer's record after a failed allocation (no GPU): its
// capacity does not outlive it.  Without a device, and for more bytes than any has,
// cudaMalloc returns an error.  Prints "ok" and exits 0 on success.
#include <cstdio>

#include "krr_internal.h"

int main() {
    krr::Ctx c;
    float *buf = nullptr;
    size_t cap = 100;  // as after an earlier call; the buffer went with the attempt to grow it
    if (krr::grow(&c, &buf, &cap, size_t(1) << 50, "test buffer") != KRR_ENOMEM) return 1;
    if (buf || cap != 0) return 2;
    if (c.last_error.find("test buffer") == std::string::npos) return 3;
    int64_t cap64 = 7;
    if (krr::grow(&c, &buf, &cap64, 7, "test buffer") != KRR_OK || cap64 != 7) return 4;  // large enough: untouched
    std::printf("ok\n");
    return 0;
}
