// Patch sizes of the field update: whole waves, one rule over all sizes.
#include <cstdio>

#include "fetdpic_internal.h"

using namespace fetdpic;

int main()
{
    for (int sms : {1, 148, 152}) {
        const long long slots = 3ll * sms;
        int before = 64;
        for (long long F = 1; F < 2500000; F += F / 997 + 1) {
            const int T = field_patch_size((int)F, sms);
            const long long patches = (F + T - 1) / T, waves = (patches + slots - 1) / slots;
            // as few waves as patches of up to 850 triangles allow, and those full but for rounding
            const long long least = (F + 850 * slots - 1) / (850 * slots);
            if (T < 64 || T > 850 || waves != least || (T > 64 && (waves * slots - patches) * (long long)T > F / 16 + waves * slots)) {
                printf("%lld triangles on %d SMs: %d a patch, %lld waves\n", F, sms, T, waves);
                return 1;
            }
            // within a wave count the patches only grow
            if (waves == 1 && T < before) { printf("%lld triangles: %d after %d\n", F, T, before); return 1; }
            if (waves == 1) before = T;
        }
    }
    return 0;
}
