// When the memory of a destroyed object goes back to the pool. Host code
// without CUDA: the runtime is a template argument, so the order of the calls
// is checked on a machine with no GPU (or only one).
#pragma once

#include <mutex>
#include <utility>
#include <vector>

namespace packsell {

// Stream-ordered memory is handed out again as soon as it is given back:
// cudaFree of it does not wait for running kernels, as it does for cudaMalloc
// memory. So an object's arrays are given back only after its own device,
// whichever device is current, has finished everything it was given; where
// that cannot be waited for (a stream of the device is being captured), the
// object stays on a list until a later call can wait.
//
// Rt: bool device(int *dev)       the current device
//     bool set_device(int dev)
//     bool wait()                 the current device has finished; false, and
//                                 no error left behind, if it cannot be waited for
//     void give_back(T *obj)      on the current device, which is obj's
template <typename T, typename Rt>
class Retired {
   public:
    void retire(int dev, T *obj, Rt rt) {
        {
            std::lock_guard<std::mutex> lock(mu_);
            late_.emplace_back(dev, obj);
        }
        flush(dev, rt);
    }

    // give back what was retired on `dev` before this call
    void flush(int dev, Rt rt) {
        std::vector<T *> mine;
        {
            std::lock_guard<std::mutex> lock(mu_);
            size_t keep = 0;
            for (auto &p : late_) {
                if (p.first == dev) mine.push_back(p.second);
                else late_[keep++] = p;
            }
            late_.resize(keep);
        }
        if (mine.empty()) return;
        int was = -1;
        const bool here = rt.device(&was) && (was == dev || rt.set_device(dev));
        const bool idle = here && rt.wait();
        if (idle)
            for (T *obj : mine) rt.give_back(obj);
        if (here && was != dev) rt.set_device(was);
        if (!idle) {
            std::lock_guard<std::mutex> lock(mu_);
            for (T *obj : mine) late_.emplace_back(dev, obj);
        }
    }

   private:
    std::mutex mu_;
    std::vector<std::pair<int, T *>> late_;
};

}  // namespace packsell
