// Host-only check of the set-up bookkeeping under threads (built with the thread sanitizer, which ends the program with an
// error when it sees a data race): every thread finds the set-up done and the value whole, whoever came first.
#include <cstdio>
#include <thread>
#include <vector>

#include "device_once.h"

int main() {
    for (int round = 0; round < 200; ++round) {
        uoe::DeviceOnce once;
        uoe::DeviceValue v;
        int wrong[4] = {};
        std::vector<std::thread> threads;
        for (int t = 0; t < 4; ++t)
            threads.emplace_back([&, t] {
                for (int dev = 0; dev < 4; ++dev) {
                    if (once.needs(dev)) once.mark(dev);
                    if (!v.has(dev)) v.set(dev, 100 + dev);
                    if (once.needs(dev) || v.get(dev) != 100 + dev) ++wrong[t];
                }
            });
        for (auto& t : threads) t.join();
        for (int w : wrong)
            if (w) return 1;
    }
    std::printf("ok\n");
    return 0;
}
