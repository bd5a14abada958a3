// Settings made once and numbers looked up once per device, for launches from any thread (host code without
// CUDA types, so that it is tested without a GPU).
#pragma once
#include <atomic>
#include <mutex>
#include <utility>
#include <vector>

namespace bp {

class OncePerDevice {
public:
    // the first call for a (device, key) runs f; every call returns after f has run
    template <class F>
    void run(int device, const void* key, F f) {
        std::lock_guard<std::mutex> lock(mu_);
        for (const auto& d : done_)
            if (d.first == device && d.second == key) return;
        f();
        done_.emplace_back(device, key);
    }

private:
    std::mutex mu_;
    std::vector<std::pair<int, const void*>> done_;
};

class NumberPerDevice {
public:
    // look_up gives a positive number, the same in every thread
    template <class F>
    int get(int device, F look_up) {
        if (device < 0 || device >= N) return look_up();
        int v = v_[device].load(std::memory_order_relaxed);
        if (v == 0) v_[device].store(v = look_up(), std::memory_order_relaxed);
        return v;
    }

private:
    static constexpr int N = 64;
    std::atomic<int> v_[N] = {};
};

}  // namespace bp
