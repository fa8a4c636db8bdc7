// gc_host.cu -- the library's host threads.
//
// Validation, the relabel plan and the packing of batches are split over the
// host's cores. Starting up to 31 threads for each of them took longer than
// many of the loops themselves (a submission of 48 graphs, an upload's six
// loops), so one pool of threads, started on first use, sleeps between them.
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <deque>
#include <exception>
#include <mutex>
#include <thread>
#include <vector>

#include "gc_internal.h"

namespace gc {
namespace {

struct Job {
  const std::function<void(int)>* f;
  int n;
  std::atomic<int> next{0};
  int inside = 0;  // threads of the pool that hold the job (under the pool's lock)
  std::exception_ptr err;
};

class Pool {
 public:
  Pool() : pid_(getpid()), threads_() {
    for (int t = 1; t < host_threads(); ++t) {
      try {
        threads_.emplace_back([this] { work(); });
      } catch (...) {
        break;  // fewer threads
      }
    }
  }
  ~Pool() {
    {
      std::lock_guard<std::mutex> lk(mu_);
      stop_ = true;
    }
    cv_.notify_all();
    for (auto& t : threads_) t.join();
  }
  bool usable() const { return getpid() == pid_; }

  void run(int n, const std::function<void(int)>& f) {
    Job job;
    job.f = &f;
    job.n = n;
    {
      std::lock_guard<std::mutex> lk(mu_);
      jobs_.push_back(&job);
    }
    const int want = std::min<int>(n - 1, (int)threads_.size());
    if (want >= (int)threads_.size()) cv_.notify_all();
    else
      for (int k = 0; k < want; ++k) cv_.notify_one();
    take(&job);
    std::unique_lock<std::mutex> lk(mu_);
    auto it = std::find(jobs_.begin(), jobs_.end(), &job);
    if (it != jobs_.end()) jobs_.erase(it);  // nobody joins it any more
    done_.wait(lk, [&] { return job.inside == 0; });
    if (job.err) std::rethrow_exception(job.err);
  }

 private:
  void take(Job* job) {
    for (int i; (i = job->next.fetch_add(1)) < job->n;) {
      try {
        (*job->f)(i);
      } catch (...) {
        std::lock_guard<std::mutex> lk(mu_);
        if (!job->err) job->err = std::current_exception();
      }
    }
  }
  void work() {
    std::unique_lock<std::mutex> lk(mu_);
    for (;;) {
      Job* job = nullptr;
      for (Job* j : jobs_)
        if (j->next.load() < j->n) {
          job = j;
          break;
        }
      if (!job) {
        if (stop_) return;
        cv_.wait(lk);
        continue;
      }
      ++job->inside;
      lk.unlock();
      take(job);
      lk.lock();
      if (--job->inside == 0) done_.notify_all();
    }
  }

  const pid_t pid_;
  std::vector<std::thread> threads_;
  std::mutex mu_;
  std::condition_variable cv_, done_;
  std::deque<Job*> jobs_;
  bool stop_ = false;
};

// The process's pool. A forked child has the object but none of its threads: it
// starts a pool of its own and leaves the parent's as it is (destroying it
// would wait for threads that the child does not have).
std::atomic<Pool*> g_pool{nullptr};

Pool* pool() {
  Pool* p = g_pool.load();
  if (p && p->usable()) return p;
  Pool* mine = new Pool();
  if (g_pool.compare_exchange_strong(p, mine)) return mine;
  delete mine;  // another thread was first
  return p;
}

struct AtExit {
  ~AtExit() {
    Pool* p = g_pool.exchange(nullptr);
    if (p && p->usable()) delete p;
  }
} g_at_exit;

}  // namespace

int host_threads() {
  static const int n = [] {
    const unsigned hw = std::thread::hardware_concurrency();
    return (int)std::min<unsigned>(hw ? hw : 1, 32);
  }();
  return n;
}

void host_run(int n, const std::function<void(int)>& f) {
  if (n > 1) {
    pool()->run(n, f);
    return;
  }
  for (int i = 0; i < n; ++i) f(i);
}

}  // namespace gc
