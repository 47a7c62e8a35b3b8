// csrc/device_once.cuh: every device's work runs, and is recorded, by itself. A kernel's attribute is set on the device that is
// current at the launch; here a table of devices stands in for the runtime.
#include <cstdio>
#include <thread>
#include <vector>

#include "device_once.cuh"

namespace {

struct Runtime {  // what the launcher asks of the CUDA runtime
    std::atomic<int> set[70] = {};
    bool fail[70] = {};
    bool launch(lgp::DeviceOnce &once, int dev) {
        if (!once.has(dev)) {
            if (fail[dev]) return false;
            set[dev].fetch_add(1);
            once.add(dev);
        }
        return set[dev].load() > 0;  // a launch on a device without the attribute is refused
    }
};

}  // namespace

int main() {
    lgp::DeviceOnce once;
    Runtime rt;
    for (int dev : {0, 1, 0, 63, 1, 5, 64, 69, 64})
        if (!rt.launch(once, dev)) return std::printf("refused on device %d\n", dev), 1;
    if (rt.set[0] != 1 || rt.set[1] != 1 || rt.set[63] != 1 || rt.set[64] != 2) return std::puts("set again or not at all"), 1;
    if (once.has(2) || once.has(-1) || once.has(64)) return std::puts("a device that was never added"), 1;
    rt.fail[7] = true;
    if (rt.launch(once, 7)) return std::puts("a failure taken for success"), 1;
    rt.fail[7] = false;
    if (!rt.launch(once, 7)) return std::puts("a failure remembered"), 1;
    lgp::DeviceOnce shared;
    std::vector<std::thread> pool;
    std::atomic<int> refused{0};
    for (int k = 0; k < 8; ++k)
        pool.emplace_back([&, k] {
            for (int i = 0; i < 6400; ++i)
                if (!rt.launch(shared, (i * 7 + k) % 64)) refused.fetch_add(1);
        });
    for (std::thread &t : pool) t.join();
    if (refused.load()) return std::puts("refused with several threads"), 1;
    std::puts("ok");
    return 0;
}
