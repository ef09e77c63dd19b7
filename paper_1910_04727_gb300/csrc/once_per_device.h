// A set-up that has to run once on every device a process uses: kernel
// attributes (the dynamic shared memory a kernel may take) belong to the device that
// was current when they were set, not to the process.
#pragma once

#include <mutex>
#include <set>

namespace fm {

class OncePerDevice {
    std::mutex mu;
    std::set<int> done;

  public:
    // f() where it has not returned on this device yet; calls from other threads wait for it.
    template <typename F>
    void run(int device, F f) {
        std::lock_guard<std::mutex> lock(mu);
        if (done.count(device)) return;
        f();
        done.insert(device);
    }
};

}  // namespace fm
