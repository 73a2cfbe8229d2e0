// Lease of the SMs for persistent (cooperative, grid-synchronised) kernels.
#pragma once
#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <mutex>
#include <vector>

#include "sw_internal.h"

// SMs that persistent (cooperative) kernels of this process hold, per device.
// A persistent launch takes its context's share of the SMs (sw_context_set_
// sm_share; all of them by default) and waits while the kernels of other
// contexts hold too many for it to fit beside them.  Grids whose shares add
// up to at most the SM count run concurrently (one CTA per SM each); others
// run one after the other, so no cooperative grid waits at a barrier for CTAs
// that cannot become resident.
//
// Leases are given in the order in which they were asked for.  The holder of a long one may
// pass a host word `yield`, which is set while other calls on the device are in flight
// (CallScope): it is to give the lease back soon and ask again, which puts it behind those
// who wait, and its kernel behind those that wait in its stream.
class SmLease {
 public:
  explicit SmLease(sw_ctx* c, volatile int* yield = nullptr)
      : dev_(c->device & 63), yield_(yield) {
    int total = 0;
    SW_CUDA(cudaDeviceGetAttribute(&total, cudaDevAttrMultiProcessorCount, c->device));
    n_ = share(c, total);
    std::unique_lock<std::mutex> lk(mu());
    State& d = state()[dev_];
    const long mine = d.next++;
    const auto ready = [&] { return d.serving == mine && d.used + n_ <= total; };
    cv().wait(lk, ready);
    ++d.serving;
    d.used += n_;
    if (yield) {
      d.yield.push_back(yield);
      ++d.yielders;
      *yield = d.calls > 1;  // one is this call
    }
    lk.unlock();
    cv().notify_all();  // the next one may fit too
  }
  ~SmLease() {
    {
      std::lock_guard<std::mutex> lk(mu());
      State& d = state()[dev_];
      d.used -= n_;
      if (yield_) {
        d.yield.erase(std::find(d.yield.begin(), d.yield.end(), yield_));
        --d.yielders;
      }
    }
    cv().notify_all();
  }
  int sms() const { return n_; }
  // The SMs a lease of this context holds, of `total`.
  static int share(const sw_ctx* c, int total) {
    const int n = (int)((long)total * c->sm_num / (c->sm_den > 0 ? c->sm_den : 1));
    return n < 1 ? 1 : (n > total ? total : n);
  }
  // A call on `device` begins or ends.
  static void call(int device, int change) {
    State& d = state()[device & 63];
    if ((d.calls += change) < 2 || change < 0 || d.yielders == 0) return;
    std::lock_guard<std::mutex> lk(mu());
    for (volatile int* y : d.yield) *y = 1;
  }

 private:
  struct State {
    int used = 0;
    long next = 0, serving = 0;  // tickets
    std::vector<volatile int*> yield;
    std::atomic<int> calls{0}, yielders{0};  // calls in flight; elements of yield
  };
  static std::mutex& mu() {
    static std::mutex m;
    return m;
  }
  static std::condition_variable& cv() {
    static std::condition_variable v;
    return v;
  }
  static State* state() {
    static State s[64];
    return s;
  }
  int dev_, n_ = 0;
  volatile int* yield_;
};
