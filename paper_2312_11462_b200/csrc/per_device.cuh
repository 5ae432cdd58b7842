// What holds for one device alone (the attributes of a kernel, how many of its clusters are resident) is asked once for
// each device of the process.  Host code without a CUDA type.
#pragma once
#include <atomic>
#include <mutex>

namespace csd {

constexpr int MAX_DEVICES = 64;

class PerDevice {
public:
    // ask() >= 0 is kept for the device; a negative answer is handed on, and the next call asks again
    template <class Ask>
    int get(int device, Ask&& ask) {
        if (device < 0 || device >= MAX_DEVICES) return ask();
        const int seen = known_[device].load(std::memory_order_acquire);
        if (seen > 0) return seen - 1;
        std::lock_guard<std::mutex> lk(mu_);
        const int again = known_[device].load(std::memory_order_relaxed);
        if (again > 0) return again - 1;
        const int answer = ask();
        if (answer >= 0) known_[device].store(answer + 1, std::memory_order_release);
        return answer;
    }

private:
    std::atomic<int> known_[MAX_DEVICES] = {};      // 0: not asked, else 1 + the answer
    std::mutex mu_;
};

}  // namespace csd
