// autotune.h -- the choice of maclab_autotune among its timings.
#pragma once

namespace maclab {
namespace autotune {

// Candidates: 0 the tile kernel; k = 1..4 the strip kernel with 4 << k rows;
// 5 the TMA-staged tile kernel; 6 the tile kernel with two steps per launch on
// clean tiles; 7 the row march; 8 the row march with two steps per pass.
constexpr int CANDIDATES = 9;
inline bool two_steps(int k) { return k == 6 || k == 8; }

struct Choice {
    int shape;     // candidate to set
    bool several;  // several steps per launch stay on
};

// ms: times of the candidates (infinite: not tried); several_ms: of several
// steps per launch.  Those go with a temporal block depth of one, so the shape
// beside them (short calls take it) is the fastest with one step per launch.
inline Choice choose(const double (&ms)[CANDIDATES], double several_ms)
{
    int best = 0, single = 0;
    for (int k = 1; k < CANDIDATES; ++k) {
        if (ms[k] < ms[best]) best = k;
        if (!two_steps(k) && ms[k] < ms[single]) single = k;
    }
    const bool several = several_ms < ms[best];
    return Choice{several ? single : best, several};
}

}  // namespace autotune
}  // namespace maclab
