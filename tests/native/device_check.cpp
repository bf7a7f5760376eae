// Host check of the per-device cache (compiled with g++ by tests/test_device_cpu.py): every device
// gets its own value, made once, also when threads ask for several devices at the same time.
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

#include "fwi_device.h"

int main()
{
    constexpr int DEV = 3;
    fwi::PerDevice<int> width;
    std::atomic<int> made[DEV] = {}, wrong{0};
    auto probe = [&](int dev) {           // devices of two kinds
        ++made[dev];
        return dev == 1 ? 8 : 16;
    };
    if (width.get(0, probe) != 16 || width.get(1, probe) != 8) return 1;   // the first device's value is not the second's
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] {
            for (int i = 0; i < 300; ++i) {
                const int dev = (i + k) % DEV;
                if (width.get(dev, probe) != (dev == 1 ? 8 : 16)) ++wrong;
            }
        });
    for (auto &x : t) x.join();
    for (const auto &m : made)
        if (m != 1) return 2;
    if (wrong) return 3;
    std::printf("device ok\n");
    return 0;
}
