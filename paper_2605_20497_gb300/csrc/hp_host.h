// hp_host.h -- host-side rules and tables without CUDA types.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace hp {

// Instances of a batch in flight when one starts: `unfinished` of them are not
// done yet (this one included), on `workers` workers.
inline int64_t batch_in_flight(int64_t workers, int64_t unfinished) { return std::min(workers, unfinished); }

// Whether an instance of a batch keeps to its one stream: its kernels that
// could run side by side only do so to use where few other streams fill the
// GPU.  Side streams against one stream, in flight: 24 power-law nets 690 and
// 726 ms (1), 396 and 411 (2), 245 and 250 (4), 204 and 187 (8), 245 and 196
// (16); eight 65k Gaussian nets 633 and 698 (1), 389 and 413 (2), 261 and 271
// (4), 224 and 211 (8); six 16k layered nets 564 and 617 (1), 231 and 241 (3),
// 147 and 148 (6); 32 random 4k nets 413 and 443 (1), 151 and 154 (4), 110 and
// 109 (8), 111 and 101 (16).
inline bool batch_one_stream(int64_t in_flight) { return in_flight >= 6; }

}  // namespace hp
