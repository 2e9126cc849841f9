// Threads of the host build's short parallel loops.  Not part of the ABI.
#pragma once

#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <cstdint>
#include <exception>
#include <mutex>
#include <thread>
#include <type_traits>
#include <vector>

namespace lc {

// Threads that live as long as one insertion of vectors and run its many short parallel loops
// (three per batch; starting 16 threads for each took 115 of 197 ms in a GPU-assisted add of 60,000
// vectors, most of them for loops with little work).  run() hands out chunks as parallel_for
// does and returns when all are done; the calling thread is thread 0.  Idle threads look for the
// next loop 2,000 times, giving way to others in between (some 0.3 ms where no one else wants the core:
// the next loop of a batch follows soon), and then sleep.
class Crew {
public:
    explicit Crew(int nt)
    {
        if (nt > 1) th_.reserve(nt - 1);                 // (may throw: no thread has started yet)
        for (int t = 1; t < nt; t++) {
            try {
                th_.emplace_back([this, t] { work(t); });
            } catch (const std::exception &) {           // no thread or no memory for one:
                break;                                   // fewer threads do the same work
            }
        }
    }
    ~Crew()
    {
        {
            std::lock_guard<std::mutex> lock(mu_);
            stop_ = true;
            job_.fetch_add(1);
        }
        cv_.notify_all();
        for (auto &x : th_) x.join();
    }
    Crew(const Crew &) = delete;
    Crew &operator=(const Crew &) = delete;

    template <class F>
    void run(int64_t n, int64_t chunk, F &&f)
    {
        if (n <= 0) return;
        chunk_ = chunk < 1 ? 1 : chunk;
        n_ = n;
        nchunks_ = (n + chunk_ - 1) / chunk_;
        if (nchunks_ == 1 || th_.empty()) {
            f((int64_t)0, n, 0);
            return;
        }
        call_ = [](void *ctx, int64_t a, int64_t b, int t) { (*static_cast<std::remove_reference_t<F> *>(ctx))(a, b, t); };
        ctx_ = &f;
        next_.store(0);
        error_ = nullptr;
        busy_.store((int)th_.size());
        {
            std::lock_guard<std::mutex> lock(mu_);
            job_.fetch_add(1);
        }
        cv_.notify_all();
        chunks(0);
        while (busy_.load() != 0) std::this_thread::yield();
        if (error_) std::rethrow_exception(error_);
    }

private:
    void chunks(int t)
    {
        try {
            for (;;) {
                const int64_t c = next_.fetch_add(1);
                if (c >= nchunks_) break;
                call_(ctx_, c * chunk_, std::min(n_, (c + 1) * chunk_), t);
            }
        } catch (...) {
            std::lock_guard<std::mutex> lock(mu_);
            if (!error_) error_ = std::current_exception();
            next_.store(nchunks_);
        }
    }
    void work(int t)
    {
        uint64_t seen = 0;
        for (;;) {
            for (int spin = 0; spin < 2000 && job_.load() == seen; spin++) std::this_thread::yield();
            if (job_.load() == seen) {
                std::unique_lock<std::mutex> lock(mu_);
                cv_.wait(lock, [&] { return job_.load() != seen; });
            }
            seen = job_.load();
            if (stop_) return;
            chunks(t);
            busy_.fetch_sub(1);
        }
    }

    std::vector<std::thread> th_;
    std::mutex mu_;
    std::condition_variable cv_;
    std::atomic<uint64_t> job_{0};               // number of the current job
    std::atomic<bool> stop_{false};
    std::atomic<int64_t> next_{0};
    std::atomic<int> busy_{0};
    std::exception_ptr error_;
    void (*call_)(void *, int64_t, int64_t, int) = nullptr;
    void *ctx_ = nullptr;
    int64_t n_ = 0, chunk_ = 1, nchunks_ = 0;
};

}  // namespace lc
