// Work done once per device: a __constant__ or __device__ symbol exists on every
// device of the process, so a table uploaded to one is not there on another.
#pragma once
#include <mutex>
#include <set>

namespace ap {

class DeviceOnce {
 public:
  // 0 if the device had it already; else what upload() returns, remembered only
  // when that is 0.  A caller returns after the upload it relies on is done,
  // whichever thread did it.
  template <class F>
  int run(int device, F&& upload) {
    std::lock_guard<std::mutex> lock(mutex_);
    if (done_.count(device)) return 0;
    const int rc = upload();
    if (rc == 0) done_.insert(device);
    return rc;
  }

 private:
  std::mutex mutex_;
  std::set<int> done_;
};

}  // namespace ap
