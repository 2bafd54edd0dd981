// ews_tuner.cuh -- the tile tuner's choice among timed trials, and what the
// choice of a batch is kept under (host code only).
#pragma once
#include <algorithm>
#include <array>
#include <cstddef>
#include <vector>

namespace ews {

// The fastest of the shapes in `cand` for a run of nt steps; cand[0] is the
// default.  time(shape, steps, &ms) times a trial; false stops the choice.
// All shapes run the same number of steps: 6, or, where the default's take
// less than half a millisecond (too short to tell shapes 5 % apart: 128 x 128
// x 64 takes 0.15 ms), as many as fill it, at most 64.  Another shape
// replaces the default only if it is 2 % faster, so shapes within timing
// noise of each other do not change from run to run.
template <typename Time>
int fastest_shape(const std::vector<int>& cand, int nt, Time time) {
    int steps = std::min(nt, 6), best = cand.front();
    float best_ms = 0.0f, ms = 0.0f;
    for (std::size_t c = 0; c < cand.size(); ++c) {
        if (!time(cand[c], steps, &ms)) return best;
        if (c == 0 && ms < 0.5f && steps < nt) {
            steps = std::min(nt, std::min(64, (int)(steps * 0.5f / std::max(ms, 1e-3f)) + 1));
            if (!time(cand[c], steps, &ms)) return best;
        }
        if (c == 0 || ms < 0.98f * best_ms) {
            best_ms = ms;
            best = cand[c];
        }
    }
    return best;
}

// What the choice between the executor and one shot after the other depends
// on: the grids with the tile shape asked for each (nx, ny, nz, shape; in any
// order), the boundary and the executor's form, the steps of the trial and the
// device it was timed on.
inline std::vector<int> batch_key(std::vector<std::array<int, 4>> shots, int boundary, int exec, int steps,
                                  int device) {
    std::sort(shots.begin(), shots.end());
    std::vector<int> key = {boundary, exec, steps, device};
    for (const auto& s : shots) key.insert(key.end(), s.begin(), s.end());
    return key;
}

}  // namespace ews
