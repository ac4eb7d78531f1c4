// Host loops shared with helper threads that the caller never waits for to start.
//
// host_parallel(n, f) calls f(i) once for every i of [0, n).  The calling thread takes the next i again and
// again; up to kHostHelpers threads of the process help, each as soon as it runs.  When all i are taken the
// caller waits only for those a helper is in the middle of.  On a host whose cores are busy (a BLAS
// pool that spins after its last call, other programs) a helper may not run for a scheduler tick, 4 ms: threads
// started and joined per copy made 24 results of 1 to 16 MB take 31 ms there, 6 ms on an idle host; with
// late helpers the caller does the work itself.
//
// Helpers wait on a semaphore, end after a second without work and are started again on demand.  Any number of threads may call at once.  f must not throw.
#pragma once
#include <semaphore.h>
#include <time.h>

#include <atomic>
#include <cerrno>
#include <cstddef>
#include <deque>
#include <memory>
#include <mutex>
#include <thread>
#include <type_traits>

namespace hostpar {

constexpr int kHostHelpers = 3;

struct Job {
  void (*call)(void* f, size_t i) = nullptr;
  void* f = nullptr;  // the caller's: used for taken indices only, and the caller outlives those
  size_t n = 0;
  std::atomic<size_t> next{0}, done{0};
  bool some() const { return next.load() < n; }
  void work() {
    for (size_t i; (i = next.fetch_add(1)) < n;) {
      call(f, i);
      done.fetch_add(1);
    }
  }
};

// The caller never blocks on a helper that is not running: it tries the lock only (also right for a process
// forked while it was held, which goes without helpers), and wakes helpers by a semaphore (a condition
// variable's notify may wait until waiters woken earlier have run).
struct Pool {
  std::mutex mu;
  sem_t wake;
  std::deque<std::shared_ptr<Job>> jobs;
  int helpers = 0;
  Pool() { sem_init(&wake, 0, 0); }

  void help() {
    for (;;) {
      std::shared_ptr<Job> j;
      {
        std::lock_guard<std::mutex> lk(mu);
        while (!jobs.empty() && !jobs.front()->some()) jobs.pop_front();
        if (!jobs.empty()) j = jobs.front();
      }
      if (j) {
        j->work();
        continue;
      }
      timespec t;
      clock_gettime(CLOCK_REALTIME, &t);
      t.tv_sec += 1;
      int r;
      while ((r = sem_timedwait(&wake, &t)) != 0 && errno == EINTR) {
      }
      if (r == 0) continue;
      std::lock_guard<std::mutex> lk(mu);
      if (!jobs.empty()) continue;
      --helpers;
      return;
    }
  }
  void post(const std::shared_ptr<Job>& j) {
    std::unique_lock<std::mutex> lk(mu, std::try_to_lock);
    if (!lk.owns_lock()) return;
    jobs.push_back(j);
    while (helpers < kHostHelpers && helpers + 1 < (int)std::thread::hardware_concurrency()) {
      std::thread(&Pool::help, this).detach();
      ++helpers;
    }
    int pending = 0;
    sem_getvalue(&wake, &pending);
    for (; pending < helpers; ++pending) sem_post(&wake);
  }
  void drop(const std::shared_ptr<Job>& j) {
    std::unique_lock<std::mutex> lk(mu, std::try_to_lock);
    if (!lk.owns_lock()) return;  // the next helper drops it
    for (auto it = jobs.begin(); it != jobs.end(); ++it)
      if (*it == j) {
        jobs.erase(it);
        return;
      }
  }
};
// never destroyed: helpers may be waiting when the process ends
inline Pool& pool() {
  static Pool* p = new Pool();
  return *p;
}

}  // namespace hostpar

template <typename F>
void host_parallel(size_t n, F&& f) {
  typedef typename std::remove_reference<F>::type Fn;
  std::shared_ptr<hostpar::Job> j;
  if (n > 1) try {
      j = std::make_shared<hostpar::Job>();
      j->call = [](void* g, size_t i) { (*static_cast<Fn*>(g))(i); };
      j->f = const_cast<void*>(static_cast<const void*>(&f));
      j->n = n;
      hostpar::pool().post(j);
    } catch (...) {  // no memory or no more threads: with the helpers there are
    }
  if (!j || j->n != n) {
    for (size_t i = 0; i < n; ++i) f(i);
    return;
  }
  j->work();
  hostpar::pool().drop(j);
  while (j->done.load(std::memory_order_acquire) < n) {  // (a yield gives the core away for a tick)
  }
}
