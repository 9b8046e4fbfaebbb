// The x-chunks of the FWI gradient's passes: which ones a pass may time (host only).
#pragma once
#include <algorithm>
#include <vector>

namespace fdgb {

// Chunks of a pass over Nx planes of `tiles` y-z tiles on `sms` multiprocessors. The first is
// what a pass too short to time them runs (and the warm-up of one that does); where it is the
// only one nothing is timed: the options name the chunk (forced > 0), or tuning is off and it
// is `untimed`.
inline std::vector<int> grad_chunks(int Nx, long long tiles, int sms, int forced, int untimed, bool tune) {
    if (forced > 0) return {std::min(forced, Nx)};
    std::vector<int> cand = {untimed};
    if (!tune) return cand;
    auto add = [&](long long c) {  // (the first is timed again after the warm-up)
        if (c >= 1 && c <= Nx && std::find(cand.begin() + 1, cand.end(), int(c)) == cand.end()) cand.push_back(int(c));
    };
    for (int c : {12, 16, 20, 32, 64}) add(c);
    for (int ctas : {3, 4, 6, 8}) {  // per SM: one and two waves
        const long long chunks = (long long)ctas * sms / tiles;
        if (chunks >= 1) add((Nx + chunks - 1) / chunks);
    }
    if (cand.size() == 1) cand.push_back(Nx);
    return cand;
}

}  // namespace fdgb
