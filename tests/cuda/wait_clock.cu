// The counted time of a wait between CTAs, for the host: a poll at each of the
// given times; returns the number of polls after which the wait gives up (0:
// never).
#include <cuda_runtime.h>

#include "acs_internal.cuh"

extern "C" int polls_until_give_up(const unsigned long long* at, int count, unsigned long long limit)
{
    unsigned long long spent = 0ull;
    for (int i = 1; i < count; ++i) {
        spent += acs::counted_wait(at[i - 1], at[i]);
        if (spent > limit) return i;
    }
    return 0;
}
