// Which of several timed launch shapes to take, where the shape also decides the order of
// sums (the batched GEMMs, batch.cu): the first one, unless a later one is faster by more than
// the noise of the timings.  Shapes that take the same time would otherwise be picked by
// that noise, and the last bits of the results with them: at n = 128, m = 4915, up to 64 images,
// pairs on 152 and on 132 SMs take 63.1-64.8 and 63.2-64.7 us, while the medians of five launches
// of one shape differ by 2 to 4 % from run to run above 50 us.
#pragma once

#include <stddef.h>

namespace tvcs {

constexpr float TUNE_GAIN = 0.05f;   // a later shape has to be faster by this part

// Launches between two events, for a matrix of rows x cols entries.  Below 50 us (2^25 entries:
// 30 to 60 us by the number of images) a single launch is timed too coarsely: the medians of
// five differed by 10 to 20 % from run to run at 10 to 20 us, those of five groups by 1 to 4 %.  Three
// groups keep the first call at a size short (n = 64, m = 1229, 40 images 3.5 -> 5.1 ms; five: 8.4);
// 12 processes gave, by launches and by groups, 3 and 2 different results at n = 64, m = 2000,
// 256 images, and at n = 128, m = 819, 40 images.
inline int tuner_launches(long long rows, long long cols) { return rows * cols <= (1LL << 25) ? 4 : 1; }

inline size_t tuned_shape(const float* t, size_t count)
{
    size_t best = 0;
    for (size_t i = 1; i < count; ++i)
        if (t[i] < (1.0f - TUNE_GAIN) * t[best]) best = i;
    return best;
}

}  // namespace tvcs
