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

// `device` is the current one while this lives, then the one before again.  Api: int get(int*)
// and int set(int), the runtime's calls.
template <typename Api> class OnDevice {
    Api api_;
    int before_ = 0, error_;
    bool changed_ = false;

public:
    OnDevice(int device, Api api = Api()) : api_(api), error_(api_.get(&before_)) {
        if (error_ || before_ == device) return;
        error_ = api_.set(device);
        changed_ = !error_;
    }
    ~OnDevice() {
        if (changed_) api_.set(before_);
    }
    OnDevice(const OnDevice&) = delete;
    OnDevice& operator=(const OnDevice&) = delete;
    int error() const { return error_; }
};

}  // namespace ptebd
