// lbm_step_graphs.h -- which of a call's steps are plain launches and which
// replay a step graph (host code that needs no CUDA header).
#pragma once

#include <stdint.h>

namespace lbm {

// Steps per captured graph, a long and a short one (even: they keep the
// ping-pong parity).  Steps launched one by one leave gaps between their two
// streams, and a small body's are shorter than their launches take the host (a
// step of 512 x 512 FP32 18.5 us so, 12.0 in a graph; 4096 x 2048 FP16 142 and
// 134); about 9 us pass between two graphs of two branches (0.5 us a step of
// 512 x 512 if all were short).
constexpr int kGraphChunk = 64, kGraphShort = 16;
constexpr int64_t kShortGraphNodes = int64_t(1) << 20;  // a step of about 20 us

// The steps of a call's next launch: a long or a short graph, or 1, a plain
// launch.  left: the call's steps still to come; queued: those it has issued;
// steps: the body's so far, with them; small: the body has fewer than
// kShortGraphNodes nodes; have_long, have_short: the graphs of the present
// parity exist.
//
// A graph takes the host 9 us a step to build, and the GPU waits for it unless
// it has work queued.  So a body's first 16 steps are plain (a new body of 701 x
// 900 FP32, 20 steps: 826 us with a graph built at once, 650 so); then a small
// body gets the short graph, and the long one with 64 steps queued (640 x 384
// FP16, a new body of 500 steps: 7.3 ms with the long one only, 6.9 so).  A
// large body's steps outlast their launches: it gets its graphs once the call
// has queued 16 plain steps (4096 x 2048: 20 steps in 3.4 ms, 3.7 with a short
// graph built first).
inline int next_steps(int64_t left, int64_t queued, int64_t steps, bool small, bool have_long, bool have_short) {
    if (left > kGraphChunk && (have_long || queued >= (small ? kGraphChunk : kGraphShort))) return kGraphChunk;
    if (left > kGraphShort && (have_short || (small ? steps : queued) >= kGraphShort)) return kGraphShort;
    return 1;
}

// The autotuners' untimed calls: after kWarmFirst and then kWarmRest steps of a
// new body, or kBatchWarm of a new batch (whose graphs take 64 steps each), the
// graphs of the parity at which the timed call starts exist, and every longer
// launch of it replays one.
constexpr int64_t kWarmFirst = 2, kWarmRest = 3 * kGraphChunk + 2, kBatchWarm = 2 * kGraphChunk + 3;

}  // namespace lbm
