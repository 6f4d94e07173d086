// DeviceOnce (csrc/device_once.h) against a fake of cudaGetDevice: the set-up runs
// once per device, again after a failure, and always where the device has no bit.
// Prints the number of wrong results.
#include <thread>
#include <vector>
#include <cstdio>

#include "device_once.h"

static thread_local int device = 0;
static thread_local cudaError_t status = cudaSuccess;
cudaError_t CUDARTAPI cudaGetDevice(int* d) {
    *d = device;
    return status;
}

int main() {
    int bad = 0, calls = 0;
    tdse::DeviceOnce once;
    auto f = [&] { ++calls; return cudaSuccess; };
    auto expect = [&](int dev, int n, cudaError_t e = cudaSuccess) {
        device = dev;
        if (once(f) != e || calls != n) ++bad;
    };
    expect(0, 1);
    expect(0, 1);
    expect(1, 2);           // a second device needs its own
    expect(0, 2);
    expect(1, 2);
    expect(63, 3);
    expect(63, 3);
    expect(64, 4);
    expect(64, 5);
    device = 2;
    if (once([] { return cudaErrorInvalidValue; }) != cudaErrorInvalidValue) ++bad;
    expect(2, 6);           // after a failure
    expect(2, 6);
    status = cudaErrorNoDevice;
    expect(2, 6, cudaErrorNoDevice);
    status = cudaSuccess;
    // several threads on devices of their own
    tdse::DeviceOnce shared;
    std::vector<int> n(8, 0);
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            device = t;
            for (int i = 0; i < 1000; ++i) shared([&] { ++n[t]; return cudaSuccess; });
        });
    for (auto& t : ts) t.join();
    for (int c : n) bad += c != 1;
    std::printf("%d\n", bad);
    return bad != 0;
}
