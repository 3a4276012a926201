// The group choice of the wave-optics calls (csrc/hpt_scratch.h) compiled with the host compiler, for the tests.
#include "hpt_scratch.h"

using namespace hpt;

extern "C" int items(long long total, size_t item_bytes, size_t most) { return group_items(total, item_bytes, most); }

// the group that an allocator of 'room' items leaves of G, and its status; 'asked': the sizes it was asked for
extern "C" int shrink(int G, int room, int other_error, int *status, int *asked, int *n_asked)
{
    int n = 0;
    *status = (int)get_group(G, [&](int g) {
        asked[n++] = g;
        return other_error ? cudaErrorInvalidValue : g <= room ? cudaSuccess : cudaErrorMemoryAllocation;
    });
    *n_asked = n;
    return G;
}
