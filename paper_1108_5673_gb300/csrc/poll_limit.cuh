// Time limit of a loop that polls without sleeping. Plain C++ too, so that the
// rule can be tested on a host.
#pragma once

#ifdef __CUDACC__
#define PWA_POLL_FN __host__ __device__ __forceinline__
#else
#define PWA_POLL_FN inline
#endif

namespace pwa {

// due() counts a poll that found nothing to do and is true at every 256th, when
// the clock is read (it is tens of cycles away); expired(now) then says whether the
// limit has passed since the first such reading. Polls that did something are not
// counted and may come anywhere in between.
struct PollLimit {
    unsigned polls = 0;
    unsigned long long first = 0;

    PWA_POLL_FN bool due() { return (++polls & 255u) == 0; }

    PWA_POLL_FN bool expired(unsigned long long now, unsigned long long limit_ns)
    {
        if (!first)
            first = now;
        return now - first > limit_ns;
    }
};

}  // namespace pwa
