// Which of a caller's vectors kernels may dereference (jac_internal.h): the
// context's own device memory, 8-byte aligned, and nothing else.
#include <cstdio>

#include "jac_internal.h"

int main()
{
    using jac::usable_in_place;
    int bad = 0;
    for (int owner = 0; owner < 3; ++owner)
        for (int device = 0; device < 3; ++device)
            for (uintptr_t at = 0x7000000000; at < 0x7000000010; ++at) {
                bad += usable_in_place(true, owner, device, at) != (owner == device && at % 8 == 0);
                bad += usable_in_place(false, owner, device, at);   // host, managed or unknown memory
            }
    std::printf(bad ? "FAIL\n" : "ok\n");
    return bad != 0;
}
