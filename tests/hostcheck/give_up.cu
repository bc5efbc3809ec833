// Host check of a split-precision call whose device wait gave up (give_up and
// plan_choice in ozaki_common.cuh): whatever width the certificate had taken,
// afterwards none is, and the plain kernel's gate is open.  Prints "cases N
// bad B".
#include <cstdio>
#include <cstring>

#include "ozaki_common.cuh"

using namespace mpdd;

int main() {
    const float thr[kMaxCand] = {1e-3f, 1e-5f, 1e-38f};
    const float margins[] = {0.0f, 1e-45f, 1e-38f, 1e-5f, 1e-3f, 1.0f, 1.0f / 0.0f};
    int cases = 0, bad = 0;
    for (int nc = 1; nc <= kMaxCand; ++nc)
        for (float d : margins) {
            SplitHeader h{};
            SplitPlan p{};
            p.dmin = &h.dmin;
            p.ncand = nc;
            memcpy(p.thr, thr, sizeof thr);
            memcpy(&h.dmin, &d, 4);
            for (int c = 0; c < nc; ++c) p.count[c] = 30 + c;
            const bool taken = plan_choice(p).c >= 0;
            give_up(&h);
            ++cases;
            if (taken != (d >= thr[nc - 1]) || plan_choice(p).c != -1 ||
                h.dmin >= p.thr[nc - 1] || h.status != MP_DD_ERR_TIMEOUT)
                ++bad;
        }
    printf("cases %d bad %d\n", cases, bad);
    return bad != 0;
}
