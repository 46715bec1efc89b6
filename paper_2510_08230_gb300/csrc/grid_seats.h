// grid_seats.h - seats of the persistent grid solvers on each device (plain
// C++, so that the queue is tested on the host).
#pragma once

#include <stdint.h>

#include <chrono>
#include <condition_variable>
#include <mutex>

namespace gk {

// One device's seats, taken in order of arrival.
class SeatPool {
public:
    // Waits until `seats` of `capacity` are free; the milliseconds it waited.
    float take(int seats, int capacity) {
        const auto t0 = std::chrono::steady_clock::now();
        std::unique_lock<std::mutex> lk(mu_);
        const uint64_t ticket = next_ticket_++;
        auto free_now = [&] { return serving_ == ticket && used_ + seats <= capacity; };
        const bool waits = !free_now();
        if (waits) freed_.wait(lk, free_now);
        used_ += seats;
        ++serving_;
        lk.unlock();
        freed_.notify_all();
        if (!waits) return 0.f;
        return std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
    }
    void give(int seats) {
        {
            std::lock_guard<std::mutex> lk(mu_);
            used_ -= seats;
        }
        freed_.notify_all();
    }

private:
    std::mutex mu_;
    std::condition_variable freed_;
    uint64_t next_ticket_ = 0, serving_ = 0;
    int used_ = 0;
};

// A pool per device ordinal (ordinals 64 apart share one).
class SeatPools {
public:
    SeatPool& of(int device) { return pools_[device >= 0 ? device % COUNT : 0]; }

private:
    static constexpr int COUNT = 64;
    SeatPool pools_[COUNT];
};

}  // namespace gk
