// Host threads of a context for its parallel host work (planning, copying
// results out).  Starting 15 threads costs about 150 us on the Grace host, more
// than most of the work they would share; waking them costs a few.
//
// One call at a time uses the workers: a call that finds them busy (another
// host thread is inside run() of the same context) does its tasks itself.
// The workers are started by the first call that wants them, at most
// kMaxWorkers and one fewer than the host's threads, and joined by the
// destructor.
#pragma once
#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <functional>
#include <mutex>
#include <system_error>
#include <thread>
#include <vector>

class RsHostPool {
 public:
  static constexpr int kMaxWorkers = 15;

  ~RsHostPool() {
    {
      std::lock_guard<std::mutex> lk(mu_);
      stop_ = true;
    }
    cv_.notify_all();
    for (auto &t : threads_) t.join();
  }

  // fn(i) for every i in [0, n), each once, on this thread and up to
  // `want - 1` workers; returns when all are done.  fn must not throw.
  void run(int n, int want, const std::function<void(int)> &fn) {
    std::unique_lock<std::mutex> use(use_, std::defer_lock);
    const int workers = std::min(want, n) > 1 && use.try_lock() ? ensure(std::min(want, n) - 1) : 0;
    if (workers < 1) {
      for (int i = 0; i < n; ++i) fn(i);
      return;
    }
    {
      std::lock_guard<std::mutex> lk(mu_);
      fn_ = &fn;
      n_ = n;
      next_.store(0, std::memory_order_relaxed);
      slots_ = workers;
      ++job_;
    }
    for (int i = 0; i < workers; ++i) cv_.notify_one();
    drain();
    std::unique_lock<std::mutex> lk(mu_);
    slots_ = 0;  // workers that have not woken yet find nothing to join
    done_.wait(lk, [&] { return inside_ == 0; });
    fn_ = nullptr;
  }

 private:
  // Started workers, at least `want` of them if the host allows (use_ held).
  int ensure(int want) {
    static const int hw = (int)std::thread::hardware_concurrency();  // a system call each time
    want = std::min({want, kMaxWorkers, std::max(hw, 1) - 1});
    while ((int)threads_.size() < want) {
      try {
        threads_.emplace_back([this] { worker(); });
      } catch (const std::exception &) {  // no thread or no memory: do with those there are
        break;
      }
    }
    return std::min(want, (int)threads_.size());
  }

  void drain() {
    for (;;) {
      const int i = next_.fetch_add(1, std::memory_order_relaxed);
      if (i >= n_) return;
      (*fn_)(i);
    }
  }

  void worker() {
    std::unique_lock<std::mutex> lk(mu_);
    uint64_t seen = 0;
    for (;;) {
      cv_.wait(lk, [&] { return stop_ || (job_ != seen && slots_ > 0); });
      if (stop_) return;
      seen = job_;
      --slots_;
      ++inside_;
      lk.unlock();
      drain();
      lk.lock();
      if (--inside_ == 0) done_.notify_one();
    }
  }

  std::mutex use_;  // held by the call that uses the workers
  std::mutex mu_;   // guards everything below but next_
  std::condition_variable cv_, done_;
  std::vector<std::thread> threads_;
  const std::function<void(int)> *fn_ = nullptr;
  std::atomic<int> next_{0};
  int n_ = 0, slots_ = 0, inside_ = 0;
  uint64_t job_ = 0;
  bool stop_ = false;
};
