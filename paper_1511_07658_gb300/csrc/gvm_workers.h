// The SPMD harnesses' threads (gvm_spmd.cu).
#pragma once

#include <atomic>
#include <chrono>
#include <condition_variable>
#include <functional>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include "gvm.h"

namespace gvm {

// The ranks' threads of a manager. Creating 15 threads, their first CUDA calls
// and their ends cost 0.8 ms a run (16 x 64 SGEMM 512^3, four steps: 0.9 of
// 4.1 ms); a kept worker is woken in some microseconds. One thread per rank of
// the runs in flight, at most; a run takes workers that no other run holds, so
// runs on disjoint ranks may overlap. An idle worker looks for work for 100 us
// and then sleeps until it is given some or the manager is shut down.
class WorkerPool {
 public:
  ~WorkerPool() {
    for (auto& w : all_) {
      {
        std::lock_guard<std::mutex> g(w->mu);
        w->stop = true;
        w->go.fetch_add(1, std::memory_order_release);
      }
      w->cv.notify_one();
      w->th.join();
    }
  }

  // fn(0) on the calling thread, fn(1) .. fn(n - 1) on workers; returns once all
  // have returned. GVM_ENOMEM, with nothing run, when a thread cannot be made.
  int run(int n, const std::function<void(int)>& fn) {
    std::vector<Worker*> mine;
    try {
      mine.reserve(n);
      std::lock_guard<std::mutex> g(mu_);
      while ((int)mine.size() < n - 1) {
        if (free_.empty()) {
          all_.reserve(all_.size() + 1);
          free_.reserve(all_.size() + 1);  // returning workers never allocates
          auto w = std::make_unique<Worker>();
          Worker* raw = w.get();
          raw->th = std::thread([raw] { raw->loop(); });
          all_.push_back(std::move(w));
          free_.push_back(raw);
        }
        mine.push_back(free_.back());
        free_.pop_back();
      }
    } catch (...) {
      give_back(mine);
      return GVM_ENOMEM;
    }
    std::atomic<int> left{n - 1};
    for (int r = 1; r < n; ++r) {
      Worker* w = mine[r - 1];
      bool asleep;
      {
        std::lock_guard<std::mutex> g(w->mu);
        w->fn = &fn;
        w->r = r;
        w->left = &left;
        w->go.fetch_add(1, std::memory_order_release);
        asleep = w->asleep;
      }
      if (asleep) w->cv.notify_one();
    }
    // An exception of a rank's ends the program, on this thread as on the others:
    // unwinding from here would leave the workers with a frame that is gone.
    [&]() noexcept { fn(0); }();
    while (left.load(std::memory_order_acquire)) std::this_thread::yield();
    give_back(mine);
    return GVM_OK;
  }

 private:
  struct Worker {
    std::thread th;
    std::mutex mu;
    std::condition_variable cv;
    std::atomic<uint32_t> go{0};  // one more for each job, and for the end
    bool asleep = false, stop = false;
    const std::function<void(int)>* fn = nullptr;
    std::atomic<int>* left = nullptr;
    int r = 0;

    void loop() {
      for (uint32_t seen = 0;; ++seen) {
        const auto t0 = std::chrono::steady_clock::now();
        while (go.load(std::memory_order_acquire) == seen &&
               std::chrono::steady_clock::now() - t0 < std::chrono::microseconds(100))
          std::this_thread::yield();
        const std::function<void(int)>* f;
        {
          std::unique_lock<std::mutex> g(mu);
          asleep = true;
          cv.wait(g, [&] { return go.load(std::memory_order_relaxed) != seen; });
          asleep = false;
          if (stop) return;
          f = fn;
        }
        (*f)(r);
        left->fetch_sub(1, std::memory_order_acq_rel);
      }
    }
  };

  void give_back(const std::vector<Worker*>& ws) {
    std::lock_guard<std::mutex> g(mu_);
    for (Worker* w : ws) free_.push_back(w);
  }

  std::mutex mu_;
  std::vector<std::unique_ptr<Worker>> all_;
  std::vector<Worker*> free_;
};

}  // namespace gvm
