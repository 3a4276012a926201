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

// walks the groups of 'total' items: how many there are, where the last begins, the items seen
extern "C" void walk(long long total, int G, long long *groups, long long *last, long long *items)
{
    *groups = *items = 0;
    (void)for_groups(total, G, [&](long long first, int n) {
        ++*groups;
        *last = first;
        *items += n;
        return first == *items - n ? cudaSuccess : cudaErrorInvalidValue;
    });
}

extern "C" int lambda_at(long long first, int f, int per) { return lambda_of(field_place(first, per), f, per); }
