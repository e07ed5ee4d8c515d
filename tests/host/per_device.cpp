// Threads that ask for a device's value while it is being found all get it
// (csrc/per_device.cuh), and it is found once per device.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>

#include "per_device.cuh"

int main() {
    lbmdem::PerDevice<int, 4> cluster;
    std::atomic<int> found{0}, wrong{0}, ready{0};
    auto find = [&] {
        ++found;
        std::this_thread::sleep_for(std::chrono::milliseconds(200));
        return 16;
    };
    std::vector<std::thread> threads;
    for (int k = 0; k < 8; ++k)
        threads.emplace_back([&] {
            ++ready;
            while (ready < 8) std::this_thread::yield();
            for (int dev : {0, 3})
                if (cluster.get(dev, find) != 16) ++wrong;
        });
    for (auto& t : threads) t.join();
    if (cluster.get(-1, find) != 0 || cluster.get(4, find) != 0) ++wrong;
    std::printf("%d wrong answers, found %d times on 2 devices\n", wrong.load(), found.load());
    return wrong || found != 2;
}
