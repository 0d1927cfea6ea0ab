// A bounded set of things that several threads use, each thing by one at a time: host
// code only, no CUDA, so that it can be checked where there is no GPU.
#pragma once

#include <condition_variable>
#include <mutex>

namespace hlf {

template <typename T, int N>
class Slots {
public:
    Slots()
    {
        for (int i = 0; i < N; ++i) free_[i] = &all_[N - 1 - i];
    }
    // One that nobody uses, the one given back last if there is a choice; waits while
    // all N are in use.
    T* take()
    {
        std::unique_lock<std::mutex> lock(mu_);
        cv_.wait(lock, [&] { return n_ > 0; });
        return free_[--n_];
    }
    void give(T* x)
    {
        {
            std::lock_guard<std::mutex> lock(mu_);
            free_[n_++] = x;
        }
        cv_.notify_one();
    }

private:
    std::mutex mu_;
    std::condition_variable cv_;
    T all_[N];
    T* free_[N];
    int n_ = N;
};

}  // namespace hlf
