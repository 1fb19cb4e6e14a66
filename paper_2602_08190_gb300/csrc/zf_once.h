// zf_once.h -- what has to be set once for each kernel on each device.
#pragma once
#include <mutex>
#include <set>
#include <utility>

namespace zf {

// A kernel's attributes (cudaFuncSetAttribute) are those of the current
// device: a process with contexts on two devices sets them twice.
class OncePerDevice {
public:
    // set() for `kernel` on `device`, until it has returned 0 (success) there.
    template <class F>
    auto operator()(int device, const void* kernel, F set) -> decltype(set()) {
        std::lock_guard<std::mutex> lock(mu_);
        const std::pair<int, const void*> key{device, kernel};
        if (done_.count(key)) return decltype(set())(0);
        const auto e = set();
        if (e == decltype(set())(0)) done_.insert(key);
        return e;
    }

private:
    std::mutex mu_;
    std::set<std::pair<int, const void*>> done_;
};

}  // namespace zf
