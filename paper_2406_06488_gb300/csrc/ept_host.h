// Host memory of the C API: copies over several cores, and the serving scheduler's sample memory.  No CUDA here.
#pragma once

#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <exception>
#include <list>
#include <memory>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

namespace ept {

// Host memory copies spread over a small pool of worker threads (the caller works
// too), used to gather pageable inputs into the pinned staging area at several times
// the bandwidth of one core.  run() returns when every byte is copied.
class HostCopier {
public:
    struct Job {
        void *dst;
        const void *src;
        size_t bytes;
    };
    // a copier of up to 8 workers, half the machine's cores; null where no thread can be started
    static std::unique_ptr<HostCopier> create() {
        const unsigned hw = std::thread::hardware_concurrency();
        std::unique_ptr<HostCopier> c(new (std::nothrow) HostCopier());
        if (!c) return c;
        try {
            for (unsigned k = std::max(1u, std::min(8u, hw / 2)); k > 0; --k)
                c->th_.emplace_back([p = c.get()] { p->worker(); });
        } catch (const std::exception &) {   // fewer workers, or none
            if (c->th_.empty()) c.reset();
        }
        return c;
    }
    ~HostCopier() {
        {
            std::lock_guard<std::mutex> lk(mu_);
            stop_ = true;
        }
        cv_.notify_all();
        for (std::thread &t : th_) t.join();
    }
    void run(const Job *jobs, size_t njobs) {
        size_t total = 0;
        for (size_t q = 0; q < njobs; ++q) total += jobs[q].bytes;
        const size_t PIECE = total >= ((size_t)32 << 20) ? (size_t)1 << 20 : (size_t)1 << 18;
        {
            std::unique_lock<std::mutex> lk(mu_);
            cv_done_.wait(lk, [this] { return active_ == 0; });   // a late worker of the last run has left
            pieces_.clear();
            for (const Job *j = jobs; j != jobs + njobs; ++j)
                for (size_t o = 0; o < j->bytes; o += PIECE)
                    pieces_.push_back({(uint8_t *)j->dst + o, (const uint8_t *)j->src + o, std::min(PIECE, j->bytes - o)});
            next_.store(0);
            remaining_.store(pieces_.size());
            ++gen_;
        }
        cv_.notify_all();
        work();
        std::unique_lock<std::mutex> lk(mu_);
        cv_done_.wait(lk, [this] { return remaining_.load() == 0 && active_ == 0; });
    }

private:
    void work() {
        const size_t n = pieces_.size();
        for (;;) {
            const size_t k = next_.fetch_add(1);
            if (k >= n) break;
            memcpy(pieces_[k].dst, pieces_[k].src, pieces_[k].bytes);
            if (remaining_.fetch_sub(1) == 1) {
                std::lock_guard<std::mutex> lk(mu_);
                cv_done_.notify_all();
            }
        }
    }
    void worker() {
        uint64_t seen = 0;
        for (;;) {
            {
                std::unique_lock<std::mutex> lk(mu_);
                cv_.wait(lk, [&] { return stop_ || gen_ != seen; });
                if (stop_) return;
                seen = gen_;
                ++active_;
            }
            work();
            {
                std::lock_guard<std::mutex> lk(mu_);
                --active_;
            }
            cv_done_.notify_all();
        }
    }
    std::vector<std::thread> th_;
    std::mutex mu_;
    std::condition_variable cv_, cv_done_;
    std::vector<Job> pieces_;
    std::atomic<size_t> next_{0}, remaining_{0};
    int active_ = 0;
    uint64_t gen_ = 0;
    bool stop_ = false;
};

// A HostCopier that several threads share: one at a time has the workers, and a thread that finds them taken
// copies by itself.  A copy too small for the workers does not ask for them, not even for a moment: a large copy
// that came just then would go to one core.
template <class Mutex>
class SharedCopier {
public:
    static constexpr size_t PARALLEL = (size_t)1 << 20;   // below, waking the workers costs what they would save
    void copy(const HostCopier::Job *jobs, size_t njobs) {
        size_t bytes = 0;
        for (size_t k = 0; k < njobs; ++k) bytes += jobs[k].bytes;
        if (bytes >= PARALLEL && copy_by_workers(jobs, njobs)) return;
        for (size_t k = 0; k < njobs; ++k) memcpy(jobs[k].dst, jobs[k].src, jobs[k].bytes);
    }

private:
    bool copy_by_workers(const HostCopier::Job *jobs, size_t njobs) {
        std::unique_lock<Mutex> lk(mu_, std::try_to_lock);
        if (!lk.owns_lock()) return false;
        if (!copier_) copier_ = HostCopier::create();
        if (!copier_) return false;
        try {
            copier_->run(jobs, njobs);
        } catch (const std::bad_alloc &) {   // no memory for the list of pieces
            return false;
        }
        return true;
    }
    Mutex mu_;
    std::unique_ptr<HostCopier> copier_;
};

struct HostBuffer {
    std::unique_ptr<float[]> data;
    size_t cap = 0;   // floats
};

// Used memory for the next requests, at most LIMIT bytes.  Copying the samples is most of a burst's time, and into
// fresh memory half of the copy is page faults: 88 MB take one core 9 ms, into used memory 5, and with the
// workers 1.3.  The oldest buffer goes when a newer one needs its place, so that requests of other sizes than
// before soon find theirs, and everything goes when nothing was taken or given for IDLE.
class HostPool {
public:
    using Clock = std::chrono::steady_clock;
    static constexpr size_t LIMIT = (size_t)256 << 20;
    static constexpr size_t SMALL = (size_t)128 << 10;   // smaller buffers are the heap's own business
    static constexpr std::chrono::milliseconds IDLE{2000};

    // Memory for `floats` values: a kept buffer of up to twice that, else a new one (data null: none to be had).
    HostBuffer take(size_t floats) {
        {
            std::lock_guard<std::mutex> lk(mu_);
            used_ = Clock::now();
            auto best = kept_.end();
            for (auto it = kept_.begin(); it != kept_.end(); ++it)
                if (it->cap >= floats && it->cap / 2 <= floats && (best == kept_.end() || it->cap < best->cap)) best = it;
            if (best != kept_.end()) {
                HostBuffer b = std::move(*best);
                kept_.erase(best);
                bytes_ -= b.cap * sizeof(float);
                return b;
            }
        }
        HostBuffer b;
        b.data.reset(new (std::nothrow) float[floats]);
        b.cap = b.data ? floats : 0;
        return b;
    }

    void give(HostBuffer b) noexcept {
        const size_t bytes = b.cap * sizeof(float);
        if (bytes < SMALL || bytes > LIMIT) return;
        std::list<HostBuffer> one, old;   // freed without the lock
        try {
            one.push_back(std::move(b));
        } catch (const std::bad_alloc &) {
            return;
        }
        std::lock_guard<std::mutex> lk(mu_);
        used_ = Clock::now();
        while (bytes_ + bytes > LIMIT) {
            bytes_ -= kept_.front().cap * sizeof(float);
            old.splice(old.end(), kept_, kept_.begin());
        }
        kept_.splice(kept_.end(), one);
        bytes_ += bytes;
    }

    bool idle(Clock::time_point now) {
        std::lock_guard<std::mutex> lk(mu_);
        return bytes_ > 0 && now - used_ >= IDLE;
    }

    void release() {
        std::list<HostBuffer> old;
        std::lock_guard<std::mutex> lk(mu_);
        old.swap(kept_);
        bytes_ = 0;
    }

    size_t bytes() {
        std::lock_guard<std::mutex> lk(mu_);
        return bytes_;
    }

private:
    std::mutex mu_;
    std::list<HostBuffer> kept_;   // oldest first
    size_t bytes_ = 0;
    Clock::time_point used_{};
};

}  // namespace ept
