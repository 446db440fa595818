// at_fit.h -- what fits on the device, asked once for a problem.
//
// The occupancy queries behind it take some tens of microseconds; their answers
// depend on a few numbers of the problem alone and are kept until one of these
// changes.  A query that failed (a negative answer) has said nothing: it stands
// for "does not fit" this time and is asked again the next.
#pragma once
#include <cstdint>
#include <cstring>

namespace atk {

struct FitCache {
    int64_t key[8] = {0};
    bool known = false;

    bool knows(const int64_t (&k)[8]) const { return known && std::memcmp(k, key, sizeof key) == 0; }

    // begins the questions for k; every answer goes through take()
    void ask(const int64_t (&k)[8])
    {
        std::memcpy(key, k, sizeof key);
        known = true;
    }
    int64_t take(int64_t answer)
    {
        if (answer < 0) known = false;
        return answer < 0 ? 0 : answer;
    }
};

} // namespace atk
