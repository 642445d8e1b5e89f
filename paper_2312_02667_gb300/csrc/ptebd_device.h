// What belongs to a device (no CUDA headers, so that the rules can be run on the CPU with
// fakes; an error is an int, 0 for none).
#pragma once
#include <map>
#include <mutex>
#include <utility>

namespace ptebd {

// Values found once per device and key, for any number of threads.  A search that failed
// is not kept: the next call searches again.
template <typename Key, typename V> class PerDevice {
    std::mutex mu_;
    std::map<std::pair<int, Key>, V> found_;

public:
    template <typename Find> V get(int device, Key key, Find&& find) {  // find(V*) -> error
        std::lock_guard<std::mutex> lock(mu_);
        const auto it = found_.find({device, key});
        if (it != found_.end()) return it->second;
        V v{};
        if (find(&v)) return V{};
        found_.emplace(std::make_pair(device, key), v);
        return v;
    }
};

}  // namespace ptebd
