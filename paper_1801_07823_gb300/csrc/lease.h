// Lease of the SMs for persistent (cooperative, grid-synchronised) kernels.
#pragma once
#include <condition_variable>
#include <mutex>

#include "sw_internal.h"

// SMs that persistent (cooperative) kernels of this process hold, per device.
// A persistent launch takes its context's share of the SMs (sw_context_set_
// sm_share; all of them by default) and waits while the kernels of other
// contexts hold too many for it to fit beside them.  Grids whose shares add
// up to at most the SM count run concurrently (one CTA per SM each); others
// run one after the other, so no cooperative grid waits at a barrier for CTAs
// that cannot become resident.
class SmLease {
 public:
  explicit SmLease(sw_ctx* c) : dev_(c->device & 63) {
    int total = 0;
    SW_CUDA(cudaDeviceGetAttribute(&total, cudaDevAttrMultiProcessorCount, c->device));
    n_ = (int)((long)total * c->sm_num / (c->sm_den > 0 ? c->sm_den : 1));
    n_ = n_ < 1 ? 1 : (n_ > total ? total : n_);
    std::unique_lock<std::mutex> lk(mu());
    cv().wait(lk, [&] { return used()[dev_] + n_ <= total; });
    used()[dev_] += n_;
  }
  ~SmLease() {
    {
      std::lock_guard<std::mutex> lk(mu());
      used()[dev_] -= n_;
    }
    cv().notify_all();
  }
  int sms() const { return n_; }

 private:
  static std::mutex& mu() {
    static std::mutex m;
    return m;
  }
  static std::condition_variable& cv() {
    static std::condition_variable v;
    return v;
  }
  static int* used() {
    static int u[64] = {0};
    return u;
  }
  int dev_, n_ = 0;
};
