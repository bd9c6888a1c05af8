// Host build of the per-device answers (device_cache.h) for the CPU test.
#include "../../paper_0707_0131_gb300/csrc/device_cache.h"

static eig::DeviceCache cache;

// answer for device when asking would give now; *asked counts
extern "C" int dc_get(int device, int now, int *asked) {
    return cache.get(device, [&] {
        ++*asked;
        return now;
    });
}
