// Rules that choose among the sweep kernels by size and shape.  Plain C++, so that
// they can be checked on the host; what each kernel is lies with the kernel.
#pragma once

#include <stdint.h>

namespace hp {

constexpr int kSMs = 152;

// Warps of a 64 x 32 window of the 26-neighbour kernel (lean.cu), by the windows of
// the launch: eight up to three windows an SM, where material points are carried and in
// the launches of an ensemble, which are not chained.  Such a launch is a chain of
// latencies -- draws, proposals, the gathers of a test -- and with twice the warps each
// goes through half as many rows; with more windows in flight the instructions count,
// and four warps issue fewer.  us per MCS, point field, four warps -> eight: 44 x 76 x 32
// (96 windows) 27.0 -> 18.6, 76 x 64 x 40 22.8 -> 15.8, 112^3 (448) 29.4 -> 23.4, but
// 128 x 128 x 64 (480) 30.0 -> 32.5; ensembles of two 48^3, grain field 22.4 -> 15.2.
inline int lean_warps(int64_t windows) { return windows <= 3 * kSMs ? 8 : 4; }

}  // namespace hp
