// hp_host.h -- host-side rules and tables without CUDA types.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <functional>
#include <unordered_map>

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

// Occupancies of kernels by block size and dynamic shared memory.  Sizes count
// in whole kilobytes: many kernels ask for bytes that follow a net's node, part
// or pin counts, and a table by bytes would grow with every net a process
// partitions (15,800 level sizes: a step call of 0.21 ms took 0.32).  So a kernel
// has at most 228 entries, and a look-up takes the same time at the process's end.
constexpr size_t SMEM_STEP = 1024;
inline size_t smem_steps(size_t bytes) { return (bytes + SMEM_STEP - 1) / SMEM_STEP; }
class OccTable {
  public:
    struct Key {
        const void *kernel;
        int device, block;
        size_t steps;
        bool operator==(const Key &o) const {
            return kernel == o.kernel && device == o.device && block == o.block && steps == o.steps;
        }
    };
    int find(const Key &k) const {   // 0: not there
        const auto it = map_.find(k);
        return it == map_.end() ? 0 : it->second;
    }
    void put(const Key &k, int occ) { map_[k] = occ; }
    size_t size() const { return map_.size(); }

  private:
    struct Hash {
        size_t operator()(const Key &k) const {
            return std::hash<const void *>()(k.kernel) ^ (k.steps * 0x9E3779B97F4A7C15ull) ^
                   ((size_t)k.block << 20) ^ ((size_t)k.device << 40);
        }
    };
    std::unordered_map<Key, int, Hash> map_;
};

}  // namespace hp
